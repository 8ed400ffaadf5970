// Building the predictor on the GPU: quantisation of W1 with the rounding error of every channel spread over the channels
// not yet rounded (GPTQ, which Section 6 of the paper names as the source of its 2-bit predictor).
//
// Per neuron (row of W1), channels in ascending order: when channel k opens a group, the group's grid (scale rounded to
// its storage type, zero-point) comes from the weights as they are then; q_k = clip(rint(w_k / s + z)),
// e_k = (w_k - s (q_k - z)) / U[k][k], and w_j <- w_j - e_k U[k][j] for j > k.  U is the upper Cholesky factor of the
// inverse Hessian of the layer's inputs, made by the caller; no U means the identity (plain rounding to nearest).
//
// Layout of the work: blocks of 64 channels in superblocks of up to 512.  k_block rounds the 64 channels of a block one after the
// other (eight lanes per neuron, its 64 weights in their registers, the 64 x 64 corner of U in shared memory) and leaves the
// 64 errors of every neuron; k_spread takes them to the later channels of the superblock, and, once the superblock is done,
// all its errors to all channels behind it (so the working copy passes through memory once per superblock), for each
// (neuron, channel) in ascending order of k.  A channel thus sees exactly the sequence of subtractions of the
// channel-by-channel procedure, each a rounded product followed by a rounded difference in double precision (no fused
// multiply-add), so the codes equal those of a plain double-precision implementation bit for bit.
// Bound by the fp64 pipe: h d^2 separate products and differences (16384 x 4096, 2.7e11: 15 ms).  Measured 23 ms of kernels (53
// before, with one thread per neuron and 16 x 1 outputs per thread, which read shared memory as often as they computed).
#include "common.cuh"

namespace tardis {
namespace {

constexpr int QB = 64;            // channels per block (divides the group size)
constexpr int NL = 8;             // lanes per neuron in k_block, QB / NL channels each
constexpr int BROWS = 16;         // neurons per CTA of k_block
constexpr int SROWS = 128;        // neurons and channels per CTA of k_spread; a thread has 8 x 4 of them
constexpr int SCOLS = 64;

template <typename T>
__global__ void k_widen(const T* __restrict__ W1, double* __restrict__ Wd, size_t count) {
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += size_t(gridDim.x) * blockDim.x)
    Wd[i] = double(to_f32<T>(W1[i]));
}

__device__ __forceinline__ double storage_round(double v, int dtype) {
  const float f = __double2float_rn(v);
  return dtype == TARDIS_F32 ? double(f) : double(__bfloat162float(__float2bfloat16_rn(f)));
}

// One block of 64 channels.  Lane l of a neuron holds channels 8 l .. 8 l + 7.  E: errors of the superblock, [channel][h].
__global__ void __launch_bounds__(BROWS * NL) k_block(double* __restrict__ Wd, const double* __restrict__ U, int h, int d, int b0, int G,
                                                      int levels, int dtype, double* __restrict__ scale64, double* __restrict__ zero64,
                                                      uint8_t* __restrict__ q, double* __restrict__ E) {
  __shared__ double2 Us[QB][4][NL];         // row i of the corner: the 16-byte pieces of a lane's 8 channels apart, lanes side by side
  __shared__ double Ud[QB];                 // its diagonal
  const int tid = threadIdx.x, l = tid & (NL - 1), r = blockIdx.x * BROWS + tid / NL;
  const int ng = d / G, g = b0 / G;
  for (int e = tid; e < QB * QB / 2; e += BROWS * NL) {
    const int i = e / (QB / 2), c2 = e - i * (QB / 2), j = c2 * 2;          // channels j, j + 1
    double2 u = make_double2(i == j ? 1.0 : 0.0, i == j + 1 ? 1.0 : 0.0);
    if (U) { const double* at = U + size_t(b0 + i) * d + b0 + j; u = make_double2(at[0], at[1]); }   // (the caller's: 8-byte aligned)
    Us[i][c2 & 3][c2 >> 2] = u;
    if (i == j) Ud[i] = u.x;
    if (i == j + 1) Ud[i] = u.y;
  }
  __syncthreads();
  const bool real = r < h;                  // (lanes of a missing neuron work on zeros: the shuffles want them)
  double w[8];
#pragma unroll
  for (int k = 0; k < 8; k += 2) {
    double2 v = make_double2(0.0, 0.0);
    if (real) v = *reinterpret_cast<const double2*>(Wd + size_t(r) * d + b0 + l * 8 + k);
    w[k] = v.x;
    w[k + 1] = v.y;
  }
  double s = 1.0, z = 0.0;
  if (b0 % G == 0) {                        // the block opens a group: its grid from the weights as they are now
    double wmin = 0.0, wmax = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) { wmin = fmin(wmin, w[k]); wmax = fmax(wmax, w[k]); }
    for (int c = QB + l; c < G && real; c += NL) {
      const double v = Wd[size_t(r) * d + b0 + c];
      wmin = fmin(wmin, v);
      wmax = fmax(wmax, v);
    }
#pragma unroll
    for (int o = 1; o < NL; o <<= 1) {
      wmin = fmin(wmin, __shfl_xor_sync(0xffffffffu, wmin, o));
      wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
    }
    s = storage_round(__ddiv_rn(__dsub_rn(wmax, wmin), double(levels)), dtype);
    if (!(s > 0.0)) s = 1.0;
    z = fmin(fmax(rint(__ddiv_rn(-wmin, s)), 0.0), double(levels));
    if (l == 0 && real) { scale64[size_t(r) * ng + g] = s; zero64[size_t(r) * ng + g] = z; }
  } else if (real) {
    s = scale64[size_t(r) * ng + g];
    z = zero64[size_t(r) * ng + g];
  }
  unsigned long long codes = 0;             // of this lane's channels, a byte each
#pragma unroll 1
  for (int lo = 0; lo < NL; ++lo) {         // channels 8 lo .. 8 lo + 7
    double err[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = lo * 8 + k;
      const double wi = __shfl_sync(0xffffffffu, w[k], lo, NL);
      const double qk = fmin(fmax(rint(__dadd_rn(__ddiv_rn(wi, s), z)), 0.0), double(levels));
      const double e = __ddiv_rn(__dsub_rn(wi, __dmul_rn(s, qk - z)), Ud[i]);
      err[k] = e;
      if (l == lo) codes |= (unsigned long long)(unsigned int)(qk) << (8 * k);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double2 u = Us[i][c][l];
        const double x = __dsub_rn(w[2 * c], __dmul_rn(e, u.x)), y = __dsub_rn(w[2 * c + 1], __dmul_rn(e, u.y));
        if (l > lo || (l == lo && 2 * c > k)) w[2 * c] = x;
        if (l > lo || (l == lo && 2 * c + 1 > k)) w[2 * c + 1] = y;
      }
    }
    if (real && l == lo) {
#pragma unroll
      for (int k = 0; k < 8; ++k) E[size_t(lo * 8 + k) * h + r] = err[k];
    }
  }
  if (real) *reinterpret_cast<unsigned long long*>(q + size_t(r) * d + b0 + l * 8) = codes;
}

// W[r][j] <- W[r][j] - e[r][i] U[k0 + i][j], i = 0 .. nk - 1 in this order (nk a multiple of 16), for the channels j0 <= j < j1 (both
// multiples of 64).  Bound by the fp64 units: per i a thread reads 12 values from shared memory for 64 fp64 instructions.  The next
// pass's values arrive by asynchronous copies meanwhile.
constexpr int SK = 16;            // channels k per pass through shared memory
__device__ __forceinline__ void copy_8_async(double* dst, const double* src, bool valid) {      // (zero where not valid)
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__global__ void __launch_bounds__(256, 2) k_spread(double* __restrict__ Wd, const double* __restrict__ U, const double* __restrict__ E,
                                                   int h, int d, int k0, int nk, int j0) {
  __shared__ __align__(16) double Es[2][SK][SROWS];
  __shared__ __align__(16) double Ut[2][SK][SCOLS];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int jb = j0 + blockIdx.x * SCOLS, r0 = blockIdx.y * SROWS;
  auto fetch = [&](int kb, int stage) {
    const int rr = threadIdx.x & (SROWS - 1), cc = threadIdx.x & (SCOLS - 1);
    const bool valid = r0 + rr < h;
    const double* es = E + size_t(kb + threadIdx.x / SROWS) * h + (valid ? r0 + rr : 0);
    const double* us = U + size_t(k0 + kb + threadIdx.x / SCOLS) * d + jb + cc;
#pragma unroll
    for (int i = 0; i < SK; i += 256 / SROWS, es += size_t(256 / SROWS) * h) copy_8_async(&Es[stage][i + threadIdx.x / SROWS][rr], es, valid);
#pragma unroll
    for (int i = 0; i < SK; i += 256 / SCOLS, us += size_t(256 / SCOLS) * d) copy_8_async(&Ut[stage][i + threadIdx.x / SCOLS][cc], us, true);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0, 0);
  double w[8][4];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int r = r0 + ty * 8 + k;
    double2 a = make_double2(0.0, 0.0), b = a;
    if (r < h) {
      const double2* src = reinterpret_cast<const double2*>(Wd + size_t(r) * d + jb + tx * 4);
      a = src[0];
      b = src[1];
    }
    w[k][0] = a.x; w[k][1] = a.y; w[k][2] = b.x; w[k][3] = b.y;
  }
  for (int kb = 0, stage = 0; kb < nk; kb += SK, stage ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                   // this pass's values are in place, the other stage has been read
    if (kb + SK < nk) fetch(kb + SK, stage ^ 1);
#pragma unroll 2
    for (int i = 0; i < SK; ++i) {
      const double2 ua = *reinterpret_cast<const double2*>(&Ut[stage][i][tx * 4]), ub = *reinterpret_cast<const double2*>(&Ut[stage][i][tx * 4 + 2]);
      const double u[4] = {ua.x, ua.y, ub.x, ub.y};
#pragma unroll
      for (int k = 0; k < 8; k += 2) {
        const double2 e2 = *reinterpret_cast<const double2*>(&Es[stage][i][ty * 8 + k]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          w[k][c] = __dsub_rn(w[k][c], __dmul_rn(e2.x, u[c]));
          w[k + 1][c] = __dsub_rn(w[k + 1][c], __dmul_rn(e2.y, u[c]));
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int r = r0 + ty * 8 + k;
    if (r < h) {
      double2* dst = reinterpret_cast<double2*>(Wd + size_t(r) * d + jb + tx * 4);
      dst[0] = make_double2(w[k][0], w[k][1]);
      dst[1] = make_double2(w[k][2], w[k][3]);
    }
  }
}

// codes into 32-bit words (channel order ascending, lowest bits first), scale into its storage type, zero-points into bytes
template <typename T>
__global__ void k_pack_out(const uint8_t* __restrict__ q, const double* __restrict__ scale64, const double* __restrict__ zero64,
                           int h, int d, int G, int bits, uint32_t* __restrict__ codes, T* __restrict__ scale, uint8_t* __restrict__ zero) {
  const int nw = d * bits / 32, ng = d / G;     // the row is one bit stream: code k holds bits [k bits, (k + 1) bits)
  const size_t words = size_t(h) * nw, groups = size_t(h) * ng;
  for (size_t e = size_t(blockIdx.x) * blockDim.x + threadIdx.x; e < words; e += size_t(gridDim.x) * blockDim.x) {
    const size_t r = e / nw;
    const int wi = int(e - r * nw);
    uint32_t word = 0u;
    const int k0 = (wi * 32) / bits, k1 = min(d - 1, (wi * 32 + 31) / bits);    // codes with a bit in this word
    for (int k = k0; k <= k1; ++k) {
      const int sh = k * bits - wi * 32;                                        // (negative: the code started in the word before)
      const uint32_t c = q[r * d + k];
      word |= sh >= 0 ? c << sh : c >> (-sh);
    }
    codes[e] = word;
  }
  for (size_t e = size_t(blockIdx.x) * blockDim.x + threadIdx.x; e < groups; e += size_t(gridDim.x) * blockDim.x) {
    scale[e] = from_f32<T>(float(scale64[e]));          // (already a value of the storage type: the conversion is exact)
    zero[e] = uint8_t(zero64[e]);
  }
}

}  // namespace

tardis_status_t launch_build_predictor(int h, int d, int dtype, const void* W1, const double* U, int bits, int G, uint32_t* codes,
                                       void* scale, uint8_t* zero, cudaStream_t s) {
  const int ng = d / G, levels = (1 << bits) - 1;
  // A group's grid is taken from weights that have seen every channel before it, so no group may reach over the end of the
  // superblock it opens in: 256 channels where groups divide that, the group itself up to 512, else single blocks.
  const int sb = 256 % G == 0 ? 256 : (G <= 512 ? G : QB);
  double *Wd = nullptr, *Eb = nullptr, *scale64 = nullptr, *zero64 = nullptr;
  uint8_t* q = nullptr;
  auto release = [&]() {
    dev_free(Wd); dev_free(Eb); dev_free(scale64); dev_free(zero64); dev_free(q);
  };
  dev_reserve(dev_room(size_t(h) * d * 8) + dev_room(size_t(h) * sb * 8) + 2 * dev_room(size_t(h) * ng * 8) + dev_room(size_t(h) * d));
  cudaError_t e = dev_malloc(&Wd, size_t(h) * d * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&Eb, size_t(h) * sb * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&scale64, size_t(h) * ng * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&zero64, size_t(h) * ng * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&q, size_t(h) * d);
  if (e != cudaSuccess) { release(); cudaGetLastError(); return TARDIS_ERR_ALLOC; }
  const size_t count = size_t(h) * d;
  if (dtype == TARDIS_F32) k_widen<float><<<2048, 256, 0, s>>>(static_cast<const float*>(W1), Wd, count);
  else k_widen<__nv_bfloat16><<<2048, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(W1), Wd, count);
  auto spread = [&](const double* errors, int k0, int nk, int j0, int j1) {   // from channels k0 .. k0 + nk - 1 to j0 .. j1 - 1
    if (U && j1 > j0) k_spread<<<dim3((j1 - j0) / SCOLS, (h + SROWS - 1) / SROWS), 256, 0, s>>>(Wd, U, errors, h, d, k0, nk, j0);
  };
  for (int s0 = 0; s0 < d && e == cudaSuccess; s0 += sb) {
    const int s1 = s0 + sb < d ? s0 + sb : d;
    for (int b0 = s0; b0 < s1; b0 += QB) {
      double* const Ebb = Eb + size_t(b0 - s0) * h;
      k_block<<<(h + BROWS - 1) / BROWS, BROWS * NL, 0, s>>>(Wd, U, h, d, b0, G, levels, dtype, scale64, zero64, q, Ebb);
      spread(Ebb, b0, QB, b0 + QB, s1);
    }
    spread(Eb, s0, s1 - s0, s1, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    if (dtype == TARDIS_F32) k_pack_out<float><<<1024, 256, 0, s>>>(q, scale64, zero64, h, d, G, bits, codes, static_cast<float*>(scale), zero);
    else k_pack_out<__nv_bfloat16><<<1024, 256, 0, s>>>(q, scale64, zero64, h, d, G, bits, codes, static_cast<__nv_bfloat16*>(scale), zero);
    e = cudaGetLastError();
  }
  const cudaError_t es = cudaStreamSynchronize(s);         // the scratch goes away with this call, whatever has been launched
  if (e == cudaSuccess) e = es;
  release();
  if (e != cudaSuccess) { set_last_error(e, "tardis_build_predictor"); return TARDIS_ERR_CUDA; }
  return TARDIS_OK;
}

}  // namespace tardis
