// Building the predictor on the GPU: quantisation of W1 with the rounding error of every channel spread over the channels
// not yet rounded (GPTQ, which Section 6 of the paper names as the source of its 2-bit predictor).
//
// Per neuron (row of W1), channels in ascending order: when channel k opens a group, the group's grid (scale rounded to
// its storage type, zero-point) comes from the weights as they are then; q_k = clip(rint(w_k / s + z)),
// e_k = (w_k - s (q_k - z)) / U[k][k], and w_j <- w_j - e_k U[k][j] for j > k.  U is the upper Cholesky factor of the
// inverse Hessian of the layer's inputs, made by the caller; no U means the identity (plain rounding to nearest).
//
// The codes are those of a plain double-precision implementation in which every product and every difference is rounded by
// itself, bit for bit.  Two ways lead to them:
//
//   k_build (bf16 layers, groups of 64 or 128 channels): one launch, a CTA takes up to 56 neurons through all channels (neurons do
//   not depend on each other, so nothing is waited for).  For 128 channels at a time the errors of all channels before them are
//   multiplied with U on the fp64 matrix instruction, weights in its accumulators; inside the 128, eight channels at a time are
//   rounded one after the other by a thread per neuron and spread over the rest by the same instruction.  Products are accumulated
//   without the intermediate rounding, so weights differ from the plain ones in the last bits.  A code can only differ where a weight
//   lies that close to a rounding boundary, so the kernel notes how close each neuron came to one; the neurons that came within
//   what the two ways can differ by (k_suspects; almost always none) are done again the plain way.
//
//   k_block and k_spread, the plain way: blocks of 64 channels in superblocks of up to 512.  k_block rounds the 64 channels of a block
//   one after the other (eight lanes per neuron, its 64 weights in their registers, the 64 x 64 corner of U in shared memory) and
//   leaves the 64 errors of every neuron; k_spread takes them to the later channels of the superblock, and, once the superblock is
//   done, all its errors to all channels behind it (so the working copy passes through memory once per superblock), for each
//   (neuron, channel) in ascending order of k.  A channel thus sees exactly the sequence of subtractions of the channel-by-channel
//   procedure, each a rounded product followed by a rounded difference (no fused multiply-add).
//
// Both are bound by the fp64 units: h d^2 / 2 multiply-adds (16384 x 4096, 1.4e11: 7.4 ms at 37 TFLOP/s), or twice as many separate
// products and differences.  16384 x 4096: 10.4 ms of kernels, 22.8 the plain way.
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace tardis {
namespace {

constexpr int QB = 64;            // channels per block (divides the group size)
constexpr int NL = 8;             // lanes per neuron in k_block, QB / NL channels each
constexpr int BROWS = 16;         // neurons per CTA of k_block
constexpr int SROWS = 128;        // neurons and channels per CTA of k_spread; a thread has 8 x 4 of them
constexpr int SCOLS = 64;

// Rows of W1 (all, or the listed ones) widened; a CTA per row in turn.
template <typename T>
__global__ void k_widen(const T* __restrict__ W1, const int* __restrict__ list, double* __restrict__ Wd, int rows, int d) {
  for (int r = blockIdx.x; r < rows; r += gridDim.x) {
    const T* const src = W1 + size_t(list ? list[r] : r) * d;
    for (int k = threadIdx.x; k < d; k += blockDim.x) Wd[size_t(r) * d + k] = double(to_f32<T>(src[k]));
  }
}

__device__ __forceinline__ double storage_round(double v, int dtype) {
  const float f = __double2float_rn(v);
  return dtype == TARDIS_F32 ? double(f) : double(__bfloat162float(__float2bfloat16_rn(f)));
}

// One block of 64 channels of h neurons: row r of Wd is neuron list[r] of scale64, zero64 and q (r itself without a list).  Lane l of a
// neuron holds channels 8 l .. 8 l + 7.  E: errors of the superblock, [channel][h].
__global__ void __launch_bounds__(BROWS * NL) k_block(double* __restrict__ Wd, const int* __restrict__ list, const double* __restrict__ U, int h,
                                                      int d, int b0, int G, int levels, int dtype, double* __restrict__ scale64,
                                                      double* __restrict__ zero64, uint8_t* __restrict__ q, double* __restrict__ E) {
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
  const int neuron = list && real ? list[r] : r;
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
    if (l == 0 && real) { scale64[size_t(neuron) * ng + g] = s; zero64[size_t(neuron) * ng + g] = z; }
  } else if (real) {
    s = scale64[size_t(neuron) * ng + g];
    z = zero64[size_t(neuron) * ng + g];
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
  if (real) *reinterpret_cast<unsigned long long*>(q + size_t(neuron) * d + b0 + l * 8) = codes;
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

// ---- k_build ------------------------------------------------------------------------------------------------------
constexpr int FB = 128;           // channels that a CTA holds in accumulators at a time: 16 per warp
constexpr int FK = 16;            // channels k per stage
constexpr int FT = 256;
constexpr int FSTAGES = 4;        // used two at a time: a barrier per 32 channels k
constexpr int FROWS = 56;         // most neurons per CTA: two CTAs of 56 on each of 148 SMs hold the 16384 of a 4096 / 16384 layer
constexpr int PROBES = 16;        // rows behind the neurons that measure how rounding errors grow (see k_suspects)

template <int MT> struct BuildCfg {               // MT: neurons per CTA in eights
  static constexpr int R = 8 * MT, ES = R + 4, US = FB + 4;           // (rows four apart modulo 16: fragments without bank conflicts)
  static constexpr int STAGE = FK * (ES + US) + FK;                   // doubles: errors [k][neuron], U [k][channel], -1 / U[k][k]
  static constexpr int SMEM = (FSTAGES * STAGE + 8 * R + 8 * R * 2) * 8;
};

__device__ __forceinline__ void copy_16_async(double* dst, const double* src, bool valid) {     // (zero where not valid)
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// How far v > 0 is from the nearest value whose bf16 is not s = bf16(float(v)); 0 where s has no ordinary neighbours.
__device__ double distance_to_other_bf16(double v, double s) {
  if (!(s > 1e-30 && s < 1e30)) return 0.0;
  const uint32_t b = __float_as_uint(float(s));
  const double below = double(__uint_as_float(b - 0x10000u)), above = double(__uint_as_float(b + 0x10000u));
  const double m0 = 0.5 * (below + s), m1 = 0.5 * (s + above);       // midpoints, themselves floats
  // a midpoint goes to the even neighbour, and so does what the rounding to float takes to the midpoint: half a step of it
  const double h0 = 0.5 * (double(__uint_as_float(__float_as_uint(float(m0)) + 1u)) - m0), h1 = 0.5 * (double(__uint_as_float(__float_as_uint(float(m1)) + 1u)) - m1);
  const double even = (b & 0x10000u) ? -1.0 : 1.0;
  return fmin(v - (m0 - even * h0), (m1 + even * h1) - v);
}

// Negated reciprocals of the diagonal of U; the largest sum of squares of a column above the diagonal (as bits: of positive numbers the
// order is the same, and no number comes out on top).  A warp takes every 32nd row of 32 columns.
__global__ void __launch_bounds__(1024) k_columns(const double* __restrict__ U, double* __restrict__ ninv, unsigned long long* __restrict__ largest, int d) {
  __shared__ double sums[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * 32 + lane, last = min(d, int(blockIdx.x + 1) * 32);
  double sum = 0.0;
#pragma unroll 16
  for (int k = warp; k < last; k += 32) {
    const double u = U[size_t(k) * d + min(j, d - 1)];
    if (k < j) sum = fma(u, u, sum);
  }
  sums[warp][lane] = sum;
  __syncthreads();
  if (warp > 0) return;
  sum = 0.0;
  for (int w = 0; w < 32; ++w) sum += sums[w][lane];
  unsigned long long top = j < d ? (unsigned long long)(__double_as_longlong(fabs(sum))) : 0ull;
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (lane == 0) atomicMax(largest, top);
  if (j < d) ninv[j] = __ddiv_rn(-1.0, U[size_t(j) * d + j]);
}

// CTA c: neurons c R .. c R + R - 1.  E: the negated errors of all its channels, [CTA][channel][R].  margin: how close (in weight) the
// neuron came to a decision that falls the other way; size: its largest weight when it was rounded; squares: the sum of its errors' squares.
// Bound by the fp64 matrix instruction, 0.72 of its rate on 16384 x 4096; U comes from L2 (67 MB per CTA), E from memory (8.6 GB in all).
// (10.8 ms with a barrier every 16 channels instead of 32; the rounding inside the blocks, a chain of six dependent fp64 operations per
// channel, is 0.6 of it.  A shorter chain for 2-bit codes, and rounding that begins while other warps still spread the eight channels
// before, need registers that are not there: 11.4.)
template <int MT>
__global__ void __launch_bounds__(FT, 2) k_build(const __nv_bfloat16* __restrict__ W1, const double* __restrict__ U, const double* __restrict__ ninv,
                                                 int h, int d, int G, int levels, double* E, double* __restrict__ scale64,
                                                 double* __restrict__ zero64, uint8_t* __restrict__ q, double* __restrict__ margin_out,
                                                 double* __restrict__ size_out, double* __restrict__ squares_out) {
  using C = BuildCfg<MT>;
  constexpr int R = C::R, ES = C::ES, US = C::US;
  extern __shared__ __align__(16) double sm[];
  double* const Wc = sm + FSTAGES * C::STAGE;       // [8][R] weights of the eight channels being rounded
  double* const ends = Wc + 8 * R;                  // [8 warps][R][2] smallest and largest weight of a warp's channels
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int r0 = blockIdx.x * R, ng = d / G;
  double* const Eg = E + size_t(blockIdx.x) * d * R;
  const int nblocks = (d + FB - 1) / FB;

  // The stages run through k = 0 .. j0 + 127 for every block of channels j0 .. j0 + 127: errors from memory up to j0, from there on
  // they are put into the stage as they arise.
  int fb = 0, fk = 0, fslot = 0;
  auto fetch = [&]() {
    if (fb < nblocks) {
      double* const st = sm + fslot * C::STAGE;
      const int j0 = fb * FB, k0 = fk * FK, cols = min(FB, d - j0);
#pragma unroll
      for (int e = tid; e < FK * FB / 2; e += FT) {
        const int k = e / (FB / 2), c = e % (FB / 2) * 2;
        copy_16_async(st + FK * ES + k * US + c, U + size_t(k0 + k) * d + j0 + (c < cols ? c : 0), c < cols);
      }
      if (k0 < j0) {
        for (int e = tid; e < FK * R / 2; e += FT) {
          const int k = e / (R / 2), c = e % (R / 2) * 2;
          copy_16_async(st + k * ES + c, Eg + size_t(k0 + k) * R + c, true);
        }
      } else if (tid < FK / 2) {
        copy_16_async(st + FK * (ES + US) + tid * 2, ninv + k0 + tid * 2, true);
      }
      if (++fk == (j0 + cols) / FK) { fk = 0; ++fb; }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    fslot = fslot == FSTAGES - 1 ? 0 : fslot + 1;
  };
  fetch();
  fetch();

  double acc[MT][4];                                // channels 16 warp + g (+ 8: elements 2, 3), neurons 8 nt + 2 t (+ 1: elements 1, 3)
  auto multiply = [&](const double* es, const double* us) {          // eight channels k
    const double* const u = us + t * US + warp * 16 + g;
    const double a0 = u[0], a1 = u[8], a2 = u[4 * US], a3 = u[4 * US + 8];
#pragma unroll
    for (int nt = 0; nt < MT; ++nt) ptx::mma_f64(acc[nt], a0, a1, a2, a3, es[t * ES + nt * 8 + g], es[(t + 4) * ES + nt * 8 + g]);
  };

  // of the thread's neuron (threads 0 .. R - 1)
  const int r = r0 + tid;
  const bool real = r < h, probe = r >= h && r < h + PROBES;
  double s = 1.0, rs = 1.0, z = 0.0, zc = 4503599627370496.0, margin = 1e300, size = 0.0;
  double squares = 0.0;                             // of the errors of neuron tid - FT / 2
  bool strange = false;

  for (int b = 0, slot = 0; b < nblocks; ++b) {
    const int j0 = b * FB, nk = (j0 + min(FB, d - j0)) / FK;
#pragma unroll
    for (int nt = 0; nt < MT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = r0 + nt * 8 + 2 * t + (i & 1), ch = j0 + warp * 16 + g + (i & 2) * 4;
        double w = 0.0;
        if (ch < d) {
          if (row < h) w = double(__bfloat162float(W1[size_t(row) * d + ch]));
          else if (row < h + PROBES) w = __popc((uint32_t(ch) * 2654435761u) & (uint32_t(row - h) * 40503u + 0x9E3779B9u)) & 1 ? 1.0 : -1.0;
        }
        acc[nt][i] = w;
      }
    for (int kt = 0; kt < nk; ++kt) {
      if ((kt & 1) == 0) {                          // (blocks have an even number of stages)
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                            // these two stages are in place, the two before have been read
        fetch();
        fetch();
      }
      double* const es = sm + slot * C::STAGE;
      const double* const us = es + FK * ES;
      slot = slot == FSTAGES - 1 ? 0 : slot + 1;
      if (kt * FK < j0) {
        multiply(es, us);
        multiply(es + 8 * ES, us + 8 * US);
        continue;
      }
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {        // eight channels, j0 + c .. j0 + c + 7
        const int c = kt * FK - j0 + half * 8, owner = c >> 4;
        const bool opens = (j0 + c) % G == 0;
        if (opens && warp >= owner && warp < owner + G / 16) {
#pragma unroll
          for (int nt = 0; nt < MT; ++nt) {
            double m[4] = {fmin(acc[nt][0], acc[nt][2]), fmax(acc[nt][0], acc[nt][2]), fmin(acc[nt][1], acc[nt][3]), fmax(acc[nt][1], acc[nt][3])};
#pragma unroll
            for (int o = 4; o < 32; o <<= 1)
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const double v = __shfl_xor_sync(0xffffffffu, m[e], o);
                m[e] = (e & 1) ? fmax(m[e], v) : fmin(m[e], v);
              }
            if (g == 0) {
              double2* const at = reinterpret_cast<double2*>(ends + (warp * R + nt * 8 + 2 * t) * 2);
              at[0] = make_double2(m[0], m[1]);
              at[1] = make_double2(m[2], m[3]);
            }
          }
        }
        if (warp == owner) {
#pragma unroll
          for (int nt = 0; nt < MT; ++nt)
            *reinterpret_cast<double2*>(Wc + g * R + nt * 8 + 2 * t) = half ? make_double2(acc[nt][2], acc[nt][3]) : make_double2(acc[nt][0], acc[nt][1]);
        }
        __syncthreads();
        if (tid < R) {
          const bool first = j0 + c == 0;           // weights as they came
          if (opens) {
            double mn = 0.0, mx = 0.0;
            for (int w = owner; w < owner + G / 16; ++w) {
              mn = fmin(mn, ends[(w * R + tid) * 2]);
              mx = fmax(mx, ends[(w * R + tid) * 2 + 1]);
            }
            const double step = __ddiv_rn(__dsub_rn(mx, mn), double(levels));
            s = storage_round(step, TARDIS_BF16);
            // (no weight but zeros, not for want of digits: the scale is 1 either way)
            if (!first && !(step == 0.0 && size == 0.0)) margin = fmin(margin, distance_to_other_bf16(step, s) * 0.5 * double(levels));
            if (!(s > 0.0)) s = 1.0;
            const double at = __ddiv_rn(-mn, s), zr = rint(at);
            if (!first && at > 0.0 && at < double(levels)) margin = fmin(margin, (0.5 - fabs(at - zr)) * s);
            z = fmin(fmax(zr, 0.0), double(levels));
            zc = 4503599627370496.0 + z;
            rs = __ddiv_rn(1.0, s);
            size = fmax(size, fmax(mx, -mn));
            if (real) {
              scale64[size_t(r) * ng + (j0 + c) / G] = s;
              zero64[size_t(r) * ng + (j0 + c) / G] = z;
            }
          }
          const double* const uc = us + half * 8 * US + c;
          const double* const ni = us + FK * US + half * 8;
          double w[8], worst = 0.0;
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = Wc[i * R + tid];
          unsigned long long codes = 0;
          // FIRST: of the neuron's first eight channels those up to the first error that is not zero are weights as they came, bf16 values
          // that tie now and then; their decisions are taken as the plain way takes them, and none of them is close.  (With the first
          // channel's alone a 4-bit layer of 8192 neurons has one done again the plain way for it.)
          auto round_eight = [&](auto first_ones) {
            constexpr bool FIRST = decltype(first_ones)::value;
            bool untouched = true;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              double v = fma(w[i], rs, z);
              if (FIRST && untouched) v = __dadd_rn(__ddiv_rn(w[i], s), z);
              // the nearest whole number in the low bits of v + 1.5 2^52; a code less the zero-point as (2^52 + q) - (2^52 + z)
              const double m = v + 6755399441055744.0, away = fabs(v - (m - 6755399441055744.0));
              const int code = min(max(__double2loint(m), 0), levels);
              strange = strange || !(fabs(v) < 1073741824.0);
              if (v > 0.0 && v < double(levels) && !(FIRST && untouched)) worst = fmax(worst, away);
              size = fmax(size, fabs(w[i]));
              const double ne = (probe ? w[i] : fma(-s, __hiloint2double(0x43300000, code) - zc, w[i])) * ni[i];
              untouched = untouched && ne == 0.0;
              es[(half * 8 + i) * ES + tid] = ne;
              Eg[size_t(j0 + c + i) * R + tid] = ne;
#pragma unroll
              for (int j = i + 1; j < 8; ++j) w[j] = fma(ne, uc[i * US + j], w[j]);
              codes |= (unsigned long long)(unsigned int)(code) << (8 * i);
            }
          };
          if (first) round_eight(std::true_type());
          else round_eight(std::false_type());
          margin = fmin(margin, (0.5 - worst) * s);
          if (real) *reinterpret_cast<unsigned long long*>(q + size_t(r) * d + j0 + c) = codes;
        }
        __syncthreads();
        // (channels that are done take part where they share a warp with ones that are not: nothing reads them any more)
        if (warp > owner || (warp == owner && half == 0)) multiply(es + half * 8 * ES, us + half * 8 * US);
        if (tid >= FT / 2 && tid < FT / 2 + R)      // (not by the threads that round: 0.2 ms of 10 in their chain)
#pragma unroll
          for (int i = 0; i < 8; ++i) { const double e = es[(half * 8 + i) * ES + tid - FT / 2]; squares = fma(e, e, squares); }
      }
    }
  }
  if (tid < R && r < h + PROBES) {
    margin_out[r] = strange ? -1.0 : margin;
    size_out[r] = strange ? 1e300 : size;
  }
  if (tid >= FT / 2 && tid < FT / 2 + R && r - FT / 2 < h + PROBES) squares_out[r - FT / 2] = squares;
}

// The neurons whose codes may not be the plain way's.  The two ways differ in the rounding of the operations, unit u = 2^-53: a weight sees up
// to 3 d of them, each of at most u times the largest sum P that it goes through.  P is bounded for any U: a part of sum e_k U[k][j] is at
// most |e| C (Cauchy and Schwarz), C the largest norm of a column above the diagonal, and with the largest weight M that was rounded
// P <= M + 2 |e| C.  With roundings of either sign that do not depend on each other, what they put into a weight stays below lambda u sqrt(d) P
// with a probability that approaches 1 as exp(-lambda^2 / 6) (the probabilistic rounding analysis of Higham and Mary, 2019).  A difference
// in one weight goes on into the later ones by the same recurrence without the rounding to codes; the probe rows have followed 16 such
// disturbances, +-1 in every channel, and A is the largest value that came of them.  lambda = 32: exp(-170).
// That P is some 45 M on a 4096 / 16384 layer and the bound 1e-11 of a weight: one layer in some 25 has a neuron that came closer than that to a
// boundary anywhere, a 4544 / 18176 layer one or two.  For up to kTightened of them the largest sum is then taken from the errors themselves
// (k_largest_sums; it is about M, and 2 to 5 ms for the plain way with a few neurons become rare).  (M in place of P misses factors whose terms
// cancel: 1.3^(j - k) above the diagonal takes sums to 1e14 and weights back to 0.1.)
constexpr int kTightened = 64;
struct Notes {                                // of k_build, behind one another in device memory
  double *ninv, *margin, *size, *squares;     // [d], [h + PROBES] each
  unsigned long long *column, *sums;          // bits of the largest column's squares; of the listed neurons' largest sums
  int *count, *list;
  static size_t bytes(int h, int d) { return (size_t(d) + 3 * (size_t(h) + PROBES) + 1 + kTightened) * 8 + (size_t(h) + 1) * 4; }
  Notes(double* at, int h, int d) : ninv(at), margin(at + d), size(margin + h + PROBES), squares(size + h + PROBES),
      column(reinterpret_cast<unsigned long long*>(squares + h + PROBES)), sums(column + 1), count(reinterpret_cast<int*>(sums + kTightened)), list(count + 1) {}
};
__device__ double growth_of(const Notes& n, int h) {
  double growth = 1.0;
  for (int p = 0; p < PROBES; ++p) growth = fmax(growth, n.size[h + p]);
  return growth;
}
__global__ void k_suspects(const Notes n, int h, double unit) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= h) return;
  const double sums = n.size[r] + 2.0 * sqrt(n.squares[r]) * sqrt(__longlong_as_double((long long)*n.column));
  if (!(n.margin[r] > unit * growth_of(n, h) * sums)) n.list[atomicAdd(n.count, 1)] = r;
}
// Block (x, y): 32 channels of the y-th neuron of the list, its weights with every error's term added in turn: a warp per 32nd of the errors,
// whose sums come first.  (One thread per channel alone waits 1.4 ms for its loads.)  E as k_build left it, R neurons per CTA.
__global__ void __launch_bounds__(1024) k_largest_sums(const Notes n, const __nv_bfloat16* __restrict__ W1, const double* __restrict__ U, const double* __restrict__ E, int d, int R) {
  __shared__ double sums[32][33];
  const int count = *n.count, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
  if (count > kTightened || int(blockIdx.y) >= count) return;
  const int r = n.list[blockIdx.y], jc = min(j, d - 1), each = (d + 31) / 32, from = warp * each, to = min(min(d, from + each), int(blockIdx.x + 1) * 32);
  const double* const e = E + size_t(r / R) * d * R + r % R;
  auto term = [&](int k) { return k < j ? e[size_t(k) * R] * U[size_t(k) * d + jc] : 0.0; };
  double sum = 0.0;
#pragma unroll 16
  for (int k = from; k < to; ++k) sum += term(k);
  sums[warp][lane] = sum;
  __syncthreads();
  double w = double(__bfloat162float(W1[size_t(r) * d + jc])), top = fabs(w);
  for (int q = 0; q < warp; ++q) w += sums[q][lane];
#pragma unroll 16
  for (int k = from; k < to; ++k) { w += term(k); top = !(fabs(w) <= top) ? fabs(w) : top; }     // (what is no number stays on top)
  unsigned long long bits = j < d ? (unsigned long long)(__double_as_longlong(top)) & 0x7fffffffffffffffull : 0ull;
  for (int o = 16; o > 0; o >>= 1) bits = max(bits, __shfl_xor_sync(0xffffffffu, bits, o));
  if (lane == 0) atomicMax(n.sums + blockIdx.y, bits);
}
__global__ void __launch_bounds__(kTightened) k_confirm(const Notes n, int h, double unit) {
  const int count = *n.count, s = threadIdx.x;
  if (count > kTightened) return;
  const int r = s < count ? n.list[s] : 0;
  const bool keep = s < count && !(n.margin[r] > unit * growth_of(n, h) * __longlong_as_double((long long)n.sums[s]));
  __syncthreads();
  if (s == 0) *n.count = 0;
  __syncthreads();
  if (keep) n.list[atomicAdd(n.count, 1)] = r;
}

struct BuildShape { int mt, ctas; };
// Neurons per CTA: as many as give every one of the 2 CTAs per SM that run together the same number of them.
BuildShape build_shape(int h, int sms) {
  const long rows = long(h) + PROBES, slots = 2L * sms, waves = (rows + slots * FROWS - 1) / (slots * FROWS);
  BuildShape s;
  s.mt = int((rows + slots * waves - 1) / (slots * waves) + 7) / 8;
  s.ctas = int((rows + 8 * s.mt - 1) / (8 * s.mt));
  return s;
}

template <int MT, typename... Args> cudaError_t launch_build(int mt, int ctas, cudaStream_t s, Args... args) {
  if constexpr (MT > FROWS / 8) { return cudaErrorInvalidValue; }
  else {
    if (mt != MT) return launch_build<MT + 1>(mt, ctas, s, args...);
    const cudaError_t e = cudaFuncSetAttribute(k_build<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, BuildCfg<MT>::SMEM);
    if (e != cudaSuccess) return e;
    k_build<MT><<<ctas, FT, BuildCfg<MT>::SMEM, s>>>(args...);
    return cudaGetLastError();
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

// k_build's conditions: bf16 layers (a float32 scale has a rounding boundary in every 1e-7 of itself, and too many neurons come close to
// one), codes of up to 4 bits (8-bit codes have 85 times as many boundaries as 2-bit ones: 8192 x 2048 5.1 ms against 4.7 the plain way,
// mostly for a few neurons done again), groups that a block of 128 channels holds, U where 16-byte copies can read it (its rows are multiples of 512 bytes).  Without U
// nothing is spread.
static bool fast_build_serves(int dtype, int bits, int G, const double* U) {
  return U && bits <= 4 && dtype == TARDIS_BF16 && (G == 64 || G == FB) && (reinterpret_cast<uintptr_t>(U) & 15u) == 0;
}

tardis_status_t launch_build_predictor(int h, int d, int dtype, const void* W1, const double* U, int bits, int G, uint32_t* codes,
                                       void* scale, uint8_t* zero, cudaStream_t s) {
  const int ng = d / G, levels = (1 << bits) - 1;
  // A group's grid is taken from weights that have seen every channel before it, so no group may reach over the end of the
  // superblock it opens in: 256 channels where groups divide that, the group itself up to 512, else single blocks.
  const int sb = 256 % G == 0 ? 256 : (G <= 512 ? G : QB);
  const bool fast = fast_build_serves(dtype, bits, G, U);
  BuildShape shape = {};
  if (fast) {
    int dev = 0, sms = 0;
    TARDIS_CUDA_TRY(cudaGetDevice(&dev));
    TARDIS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    shape = build_shape(h, sms);
  }
  // the plain way's working copy and, before it, the errors of k_build share their memory
  const size_t wd_bytes = fast ? size_t(shape.ctas) * 8 * shape.mt * d * 8 : size_t(h) * d * 8;
  const size_t notes_bytes = fast ? Notes::bytes(h, d) : 0;
  double *Wd = nullptr, *Eb = nullptr, *scale64 = nullptr, *zero64 = nullptr, *notes = nullptr;
  uint8_t* q = nullptr;
  auto release = [&]() {
    dev_free(Wd); dev_free(Eb); dev_free(scale64); dev_free(zero64); dev_free(q); dev_free(notes);
  };
  dev_reserve(dev_room(wd_bytes) + dev_room(size_t(h) * sb * 8) + 2 * dev_room(size_t(h) * ng * 8) + dev_room(size_t(h) * d) +
              (fast ? dev_room(notes_bytes) : 0));
  cudaError_t e = dev_malloc(&Wd, wd_bytes);
  if (e == cudaSuccess) e = dev_malloc(&Eb, size_t(h) * sb * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&scale64, size_t(h) * ng * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&zero64, size_t(h) * ng * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&q, size_t(h) * d);
  if (e == cudaSuccess && fast) e = dev_malloc(&notes, notes_bytes);
  if (e != cudaSuccess) { release(); cudaGetLastError(); return TARDIS_ERR_ALLOC; }
  const int* list = nullptr;                               // the neurons that are done the plain way (null: all)
  int rows = h;
  if (fast) {
    const Notes n(notes, h, d);
    list = n.list;
    const double unit = 32.0 * 1.1102230246251565e-16 * sqrt(double(d));
    e = cudaMemsetAsync(n.column, 0, reinterpret_cast<char*>(n.list) - reinterpret_cast<char*>(n.column), s);
    k_columns<<<(d + 31) / 32, 1024, 0, s>>>(U, n.ninv, n.column, d);
    if (e == cudaSuccess)
      e = launch_build<1>(shape.mt, shape.ctas, s, static_cast<const __nv_bfloat16*>(W1), U, static_cast<const double*>(n.ninv), h, d, G, levels, Wd,
                          scale64, zero64, q, n.margin, n.size, n.squares);
    k_suspects<<<(h + 255) / 256, 256, 0, s>>>(n, h, unit);
    k_largest_sums<<<dim3((d + 31) / 32, kTightened), 1024, 0, s>>>(n, static_cast<const __nv_bfloat16*>(W1), U, Wd, d, 8 * shape.mt);
    k_confirm<<<1, kTightened, 0, s>>>(n, h, unit);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&rows, n.count, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  if (e == cudaSuccess && rows > 0) {
    if (dtype == TARDIS_F32) k_widen<float><<<2048, 256, 0, s>>>(static_cast<const float*>(W1), list, Wd, rows, d);
    else k_widen<__nv_bfloat16><<<2048, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(W1), list, Wd, rows, d);
    auto spread = [&](const double* errors, int k0, int nk, int j0, int j1) {   // from channels k0 .. k0 + nk - 1 to j0 .. j1 - 1
      if (U && j1 > j0) k_spread<<<dim3((j1 - j0) / SCOLS, (rows + SROWS - 1) / SROWS), 256, 0, s>>>(Wd, U, errors, rows, d, k0, nk, j0);
    };
    for (int s0 = 0; s0 < d && e == cudaSuccess; s0 += sb) {
      const int s1 = s0 + sb < d ? s0 + sb : d;
      for (int b0 = s0; b0 < s1; b0 += QB) {
        double* const Ebb = Eb + size_t(b0 - s0) * rows;
        k_block<<<(rows + BROWS - 1) / BROWS, BROWS * NL, 0, s>>>(Wd, list, U, rows, d, b0, G, levels, dtype, scale64, zero64, q, Ebb);
        spread(Ebb, b0, QB, b0 + QB, s1);
      }
      spread(Eb, s0, s1 - s0, s1, d);
      e = cudaGetLastError();
    }
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
