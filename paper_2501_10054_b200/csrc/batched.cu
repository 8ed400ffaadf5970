// Batched / prefill form of the online path (Section 5.4) for bf16 layers: every step is a dense product on
// the tcgen05 tensor cores (gemm.cu) or a light elementwise pass.
//
// For a chunk of up to kChunk tokens X[n, d]:
//   1. fast predictor scores  Zhat = X What^T + b1, What = s (q - zp) (Section 5.3).  What needs up to 10 significant
//      bits (13 with 4-bit codes), so it is held as an exact sum of two bf16 matrices (hi + lo).  With 2-bit codes lo is
//      zero wherever |q - zp| <= 2, which is every group whose weights have both signs: the fold notes which 128-row
//      tiles need lo at all, and the score GEMM leaves it out for the others (half of its work; 16384 prompt tokens of a
//      4096 / 16384 layer 10.1 -> 9.2 ms, 32 tokens of an 8192 / 32768 layer 522 -> 445 us).  Its epilogue turns the scores into flag words (they are stored only for the debug
//      capture).  Products are exact, the fp32 accumulation is not: a score within
//      tau(t, j) = kEps * (2^bits - 1) max_g s[j,g] * |x_t|_1 of a range end is queued by the epilogue and
//      re-evaluated in fp64 from the packed codes (k_recheck), so the flags are the exact ones;
//   2. result fixing          Delta = flag .* (GELU(Z) - a Z - c), Z = X W1^T + b1   (GEMM with that epilogue, bf16);
//   3. output                 y = bf16(X W_f^T + b_f + Delta W2^T), the speculative product and the corrections over all neurons in one
//      GEMM (with independent ~10 % flags the union over >= 64 tokens is practically every neuron, which is why
//      the paper expects little gain for prompt-heavy requests).
#include <vector>

#include "common.cuh"
#include "exact.cuh"
#include "gemm.cuh"

namespace tardis {
namespace bat {

// Tokens per pass (the scratch is sized for this).  With 2048 the big products have 16 x 64 tiles = 6.9 waves of
// 148 CTAs; 1024-token chunks lost 15 % of the time to their last, partial wave.
constexpr int kChunk = 2048;
constexpr int kSplitTokens = 128;            // calls of up to this many split their output product, whose parts meet in an fp32 array
constexpr int kChunkCapture = 1024;          // ... while the debug capture is on (the score buffer holds that many)
constexpr float kEps = 7.62939453125e-6f;    // 2^-17: relative accumulation-error allowance of the fast scores
// neurons per token that can queue for re-evaluation: a sixteenth, some ten times what narrow ranges of a 4096 / 16384 layer need (the
// allowance grows with d, the spread of the scores with its root: a fixed number would be too small for the widest layers)
__host__ __device__ constexpr int max_recheck(int h) { return h / 16 > 512 ? h / 16 : 512; }

struct State {
  __nv_bfloat16 *Wf, *W2, *What_hi, *What_lo;     // [d,d], [d,h], [h,d], [h,d]
  float* smaxrow;                                  // [h] largest group scale of a neuron
  uint32_t* lo_used;                               // [h / 128 rounded up] bit 0: What_lo is not zero in those rows; bit 1: some |q - zp| > 2
  float *zhat, *yacc, *x1;                         // [kChunkCapture,h] (scores for the capture; fold temporary), [kSplitTokens,d], [kChunk]
  __nv_bfloat16* delta;                            // [kChunk,h]
  uint32_t* bitmap;                                // [kChunk,h/32]
  uint32_t* rlist;                                 // [kChunk][max_recheck(h)] neurons of a token to re-evaluate
  unsigned int* rcount;                            // [kChunk] how many (more than the queue holds: every neuron is re-evaluated)
  size_t bytes_state, bytes_scratch;
};

// ---- set-up ---------------------------------------------------------------------------------------------
// What = s (q - zp) split exactly into hi = bf16(What) and lo = What - hi (at most 2 significant bits left).
// A row per CTA; a thread takes 8 channels (one group: groups are multiples of 16 channels) and writes 16 bytes of either matrix.
__global__ void k_dequant_split(const uint32_t* __restrict__ codes, const __nv_bfloat16* __restrict__ scale,
                                const uint8_t* __restrict__ zero, __nv_bfloat16* __restrict__ hi,
                                __nv_bfloat16* __restrict__ lo, float* __restrict__ smaxrow, uint32_t* __restrict__ lo_used, int d, int G, int bits) {
  __shared__ float wmax[8];
  uint32_t notes = 0u;                          // of this thread's values: 1 one has a second term, 2 one has |q - zp| > 2 (3 s may well be a bf16 value)
  float smax = 0.f;
  const int j = blockIdx.x, ng = d / G;
  const uint32_t* row = codes + size_t(j) * (size_t(d) * bits / 32);
  for (int k0 = threadIdx.x * 8; k0 < d; k0 += blockDim.x * 8) {
    const int g = k0 / G;
    const float s = __bfloat162float(scale[size_t(j) * ng + g]), zp = float(zero[size_t(j) * ng + g]);
    smax = fmaxf(smax, fabsf(s));
    __nv_bfloat162 h[4], l[4];
    // (2- and 4-bit codes of eight channels lie in one word, and k0 is a multiple of 8)
    const bool whole = bits == 2 || bits == 4;
    const uint32_t word = whole ? row[k0 * bits >> 5] >> (k0 * bits & 31) : 0u, mask = (1u << bits) - 1u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float v[2], t[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float m = float(whole ? (word >> (bits * (2 * q + e))) & mask : stream_code(row, k0 + 2 * q + e, bits)) - zp;
        v[e] = s * m;                                                      // exact: 8-bit significand times |int| <= 15
        t[e] = __bfloat162float(__float2bfloat16_rn(v[e]));
        notes |= (v[e] != t[e] ? 1u : 0u) | (fabsf(m) > 2.f ? 2u : 0u);
      }
      h[q] = __floats2bfloat162_rn(t[0], t[1]);
      l[q] = __floats2bfloat162_rn(v[0] - t[0], v[1] - t[1]);
    }
    *reinterpret_cast<uint4*>(hi + size_t(j) * d + k0) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + size_t(j) * d + k0) = *reinterpret_cast<const uint4*>(l);
  }
  notes = __reduce_or_sync(0xffffffffu, notes);
  if (notes && (threadIdx.x & 31) == 0) atomicOr(&lo_used[j >> 7], notes);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = smax;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (blockDim.x >> 5); ++w) smax = fmaxf(smax, wmax[w]);
    smaxrow[j] = smax;
  }
}

// ---- per-chunk passes -----------------------------------------------------------------------------------
// |x_t|_1 (inf when the token holds a non-finite value: every neuron of it is then flagged)
__global__ void k_xnorm(const __nv_bfloat16* __restrict__ x, int d, float* __restrict__ x1) {
  __shared__ float red[32];
  const int t = blockIdx.x;
  float s = 0.f;
  bool bad = false;
  for (int k = threadIdx.x * 8; k < d; k += blockDim.x * 8) {          // (d is a multiple of 8)
    const uint4 v = *reinterpret_cast<const uint4*>(x + size_t(t) * d + k);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float a = fabsf(__uint_as_float(w[q] << 16)), b = fabsf(__uint_as_float(w[q] & 0xffff0000u));
      bad |= !(a <= 3.0e38f) || !(b <= 3.0e38f);
      s += a + b;
    }
  }
  if (bad) s = __int_as_float(0x7f800000);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float tot = 0.f;
    for (int w = 0; w < (blockDim.x + 31) / 32; ++w) tot += red[w];
    x1[t] = tot;
  }
}

// A CTA per token: the exact fp64 scores of its queued neurons (one warp each, from the packed codes) decide their flags; then the
// token's flags are counted.  Where more neurons wanted to queue than fit, all are re-evaluated (one such token among 200 of
// 4096 / 16384: 9 ms; each settled by the thread that met it, in the product's epilogue: 19 ms).  The token is widened to fp64 once, in shared memory: with a conversion per product these, at 16 per
// clock and SM, were the bound (2048 tokens on 4096 / 16384: 51 us, 93 before with the count as a kernel of its own).
// WIDTH: bits per code where 32 is a multiple of it, else 0.  STAGED: false for tokens that do not fit in shared memory.
template <int WIDTH, bool STAGED>
__global__ void __launch_bounds__(256) k_recheck(const uint32_t* __restrict__ rlist, const unsigned int* __restrict__ rcount, const uint32_t* __restrict__ codes,
                                                 const __nv_bfloat16* __restrict__ scale, const uint8_t* __restrict__ zero, const float* __restrict__ b1,
                                                 const float* __restrict__ lo, const float* __restrict__ hi, const __nv_bfloat16* __restrict__ x, int d, int h,
                                                 int G, int bits, uint32_t* __restrict__ bitmap, float* __restrict__ zhat, unsigned long long* counters) {
  extern __shared__ double xd[];                           // channel c of unit u (16 channels) at c (d / 16 + 1) + u: the lanes' units side by side
  __shared__ unsigned int flagged;
  const int t = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned int queued = rcount[t];
  const unsigned int most = max_recheck(h);
  const bool all = queued > most;
  const unsigned int total = all ? (unsigned int)h : queued;
  const __nv_bfloat16* const xt = x + size_t(t) * d;
  const int nw = d / 16;
  auto xv = [&](int u, int c) { return STAGED ? xd[c * (nw + 1) + u] : double(__bfloat162float(xt[u * 16 + c])); };
  if (threadIdx.x == 0) flagged = 0u;
  if (STAGED && total > 0)
    for (int u = threadIdx.x; u < nw; u += blockDim.x) {
      const uint4 a = *reinterpret_cast<const uint4*>(xt + u * 16), b = *reinterpret_cast<const uint4*>(xt + u * 16 + 8);
      const uint32_t v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        xd[2 * c * (nw + 1) + u] = double(__uint_as_float(v[c] << 16));
        xd[(2 * c + 1) * (nw + 1) + u] = double(__uint_as_float(v[c] & 0xffff0000u));
      }
    }
  __syncthreads();
  const int ng = d / G;
  for (unsigned int e = warp; e < total; e += 8) {
    const int j = all ? int(e) : int(rlist[size_t(t) * most + e]);
    const uint32_t* const row = codes + size_t(j) * (size_t(d) * bits / 32);
    double z = 0.0;
    // units of 16 channels (all of one group), four at a time: their loads go out before the first is used, since waiting for them
    // is most of what a warp does here
    for (int u0 = lane; u0 < nw; u0 += 128) {
      uint32_t w[4][WIDTH ? WIDTH / 2 : 1];
      __nv_bfloat16 sc[4];
      uint8_t zr[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int u = u0 + 32 * v;
        if (u < nw) {
          sc[v] = scale[size_t(j) * ng + u * 16 / G];
          zr[v] = zero[size_t(j) * ng + u * 16 / G];
          if (WIDTH) {
#pragma unroll
            for (int q = 0; q < WIDTH / 2; ++q) w[v][q] = row[u * (WIDTH / 2) + q];
          }
        }
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int u = u0 + 32 * v;
        if (u >= nw) break;
        const double zp = 4503599627370496.0 + double(zr[v]);
        double p0 = 0.0, p1 = 0.0;
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const uint32_t q0 = WIDTH ? (w[v][c * WIDTH / 32] >> (c * WIDTH % 32)) & ((1u << WIDTH) - 1u) : stream_code(row, u * 16 + c, bits);
          const uint32_t q1 = WIDTH ? (w[v][(c + 1) * WIDTH / 32] >> ((c + 1) * WIDTH % 32)) & ((1u << WIDTH) - 1u) : stream_code(row, u * 16 + c + 1, bits);
          // (2^52 + q) - (2^52 + zp): the code less the zero-point without a conversion
          p0 += (__hiloint2double(0x43300000, int(q0)) - zp) * xv(u, c);
          p1 += (__hiloint2double(0x43300000, int(q1)) - zp) * xv(u, c + 1);
        }
        z += double(__bfloat162float(sc[v])) * (p0 + p1);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    z += double(b1[j]);
    if (lane == 0) {
      const bool inside = (double(lo[j]) <= z) && (z < double(hi[j]));
      uint32_t* wp = bitmap + size_t(t) * (h / 32) + (j >> 5);
      if (inside) atomicAnd(wp, ~(1u << (j & 31)));
      else atomicOr(wp, 1u << (j & 31));
      if (zhat) zhat[size_t(t) * h + j] = float(z);
    }
  }
  __threadfence_block();
  __syncthreads();
  unsigned int c = 0;
  for (int w = threadIdx.x; w < h / 32; w += blockDim.x) c += __popc(__ldcg(bitmap + size_t(t) * (h / 32) + w));
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) atomicAdd(&flagged, c);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (flagged) {
      atomicAdd(&counters[CTR_FLAGGED_TOTAL], (unsigned long long)flagged);
      atomicMax(&counters[CTR_FLAGGED_MAX], (unsigned long long)flagged);
    }
    if (total) atomicAdd(&counters[CTR_RECHECKS], (unsigned long long)total);
  }
}

__global__ void k_round_store(const float* __restrict__ yacc, __nv_bfloat16* __restrict__ y, size_t count) {
  const size_t e = (size_t(blockIdx.x) * blockDim.x + threadIdx.x) * 4;
  if (e + 3 < count) {
    const float4 v = *reinterpret_cast<const float4*>(yacc + e);
    __nv_bfloat162 o[2] = {__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
    *reinterpret_cast<uint2*>(y + e) = *reinterpret_cast<const uint2*>(o);
  } else {
    for (size_t i = e; i < count; ++i) y[i] = __float2bfloat16_rn(yacc[i]);
  }
}

__global__ void k_capture(const uint32_t* __restrict__ bitmap, const float* __restrict__ zhat, const float* __restrict__ x1,
                          int n, int h, uint32_t* __restrict__ dbg_bitmap, double* __restrict__ dbg_scores) {
  const size_t e = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= size_t(n) * h) return;
  if (dbg_scores) {
    const int t = int(e / h);
    dbg_scores[e] = (x1[t] <= 3.0e38f) ? double(zhat[e]) : __longlong_as_double(0x7ff8000000000000ll);
  }
  if (dbg_bitmap && e < size_t(n) * (h / 32)) dbg_bitmap[e] = bitmap[e];
}

}  // namespace bat

using namespace bat;

namespace {
struct Req { void** p; size_t bytes; bool scratch; };
struct Requests { Req r[13]; };
Requests requests(State* S, int d, int h) {
  const size_t hd = size_t(h) * d;
  const Requests all = {{
      {reinterpret_cast<void**>(&S->Wf), size_t(d) * d * 2, false}, {reinterpret_cast<void**>(&S->W2), hd * 2, false},
      {reinterpret_cast<void**>(&S->What_hi), hd * 2, false},       {reinterpret_cast<void**>(&S->What_lo), hd * 2, false},
      {reinterpret_cast<void**>(&S->smaxrow), size_t(h) * 4, false}, {reinterpret_cast<void**>(&S->lo_used), size_t((h + 127) / 128) * 4, false},
      {reinterpret_cast<void**>(&S->zhat), size_t(kChunkCapture) * h * 4, true}, {reinterpret_cast<void**>(&S->yacc), size_t(kSplitTokens) * d * 4, true},
      {reinterpret_cast<void**>(&S->x1), size_t(kChunk) * 4, true},       {reinterpret_cast<void**>(&S->delta), size_t(kChunk) * h * 2, true},
      {reinterpret_cast<void**>(&S->bitmap), size_t(kChunk) * (h / 32) * 4, true},
      {reinterpret_cast<void**>(&S->rlist), size_t(kChunk) * max_recheck(h) * 4, true},
      {reinterpret_cast<void**>(&S->rcount), size_t(kChunk) * 4, true}}};
  return all;
}
bool served(const Handle* H) { return H->dtype == TARDIS_BF16 && H->d % 8 == 0 && H->h % 32 == 0; }
}  // namespace

size_t batched_room(const Handle* H) {
  if (!served(H)) return 0;
  State S = {};
  size_t room = few_room(H);
  for (const Req& r : requests(&S, H->d, H->h).r) room += dev_room(r.bytes);
  return room;
}

tardis_status_t batched_prepare(Handle* H) {
  H->bstate = nullptr;
  const int d = H->d, h = H->h;
  if (!served(H)) return TARDIS_OK;
  State* S = new (std::nothrow) State();
  if (!S) return TARDIS_ERR_ALLOC;
  memset(S, 0, sizeof(*S));
  H->bstate = S;
  const size_t hd = size_t(h) * d;
  for (const Req& r : requests(S, d, h).r) {
    cudaError_t e = dev_malloc(r.p, r.bytes);
    if (e != cudaSuccess) { set_last_error(e, "cudaMalloc"); cudaGetLastError(); batched_release(H); return TARDIS_ERR_ALLOC; }
    (r.scratch ? S->bytes_scratch : S->bytes_state) += r.bytes;
  }
  H->bytes_folded += size_t(d) * d * 2;
  H->bytes_w2t += hd * 2;                       // second copy of W2 (original orientation)
  H->bytes_predictor += 2 * hd * 2 + size_t(h) * 4 + size_t((h + 127) / 128) * 4;
  H->bytes_scratch += S->bytes_scratch;
  const tardis_status_t st = few_prepare(H);
  if (st != TARDIS_OK) batched_release(H);
  return st;
}

// a_j W1[j][k] in fp32, transposed to [k][j] and split into bf16 hi + lo (16 significant bits together); 64 x 64 at a time, two elements
// per access (h and d are even; 16384 x 4096: 75 us, 172 one by one)
__global__ void __launch_bounds__(256) k_scale_transpose_split(const uint32_t* __restrict__ W1, const float* __restrict__ a,
                                                               uint32_t* __restrict__ hi, uint32_t* __restrict__ lo, int h, int d) {
  __shared__ uint32_t tile[64][33];                                   // [neuron][channel pair]
  const int k0 = blockIdx.x * 64, j0 = blockIdx.y * 64, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int r = warp; r < 64; r += 8)
    if (j0 + r < h && k0 + 2 * lane < d) tile[r][lane] = W1[(size_t(j0 + r) * d + k0) / 2 + lane];
  __syncthreads();
  const int j = j0 + 2 * lane;
  if (j >= h) return;
  const float a0 = a[j], a1 = a[j + 1];
#pragma unroll
  for (int p = warp; p < 32; p += 8) {                                // channels k0 + 2 p, k0 + 2 p + 1 of neurons j, j + 1
    if (k0 + 2 * p >= d) continue;
    const uint32_t w0 = tile[2 * lane][p], w1 = tile[2 * lane + 1][p];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float v0 = a0 * __uint_as_float(c ? w0 & 0xffff0000u : w0 << 16), v1 = a1 * __uint_as_float(c ? w1 & 0xffff0000u : w1 << 16);
      const __nv_bfloat162 top = __floats2bfloat162_rn(v0, v1);
      const __nv_bfloat162 rest = __floats2bfloat162_rn(v0 - __bfloat162float(top.x), v1 - __bfloat162float(top.y));
      const size_t at = (size_t(k0 + 2 * p + c) * h + j) / 2;
      hi[at] = *reinterpret_cast<const uint32_t*>(&top);
      lo[at] = *reinterpret_cast<const uint32_t*>(&rest);
    }
  }
}

// rows [i0, i0 + rows) of W_f (fp32) rounded once to bf16 and stored as C[k][i]
__global__ void k_store_folded(const float* __restrict__ Wf32, __nv_bfloat16* __restrict__ C, int i0, int rows, int d) {
  __shared__ float tile[32][33];
  const int k0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int ii = r0 + r, k = k0 + threadIdx.x;
    if (ii < rows && k < d) tile[r][threadIdx.x] = Wf32[size_t(ii) * d + k];
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, ii = r0 + threadIdx.x;
    if (ii < rows && k < d) C[size_t(k) * d + i0 + ii] = __float2bfloat16_rn(tile[threadIdx.x][r]);
  }
}

// Constant folding (Section 5.2) on the tensor cores: W_f = W2 (diag(a) W1), with diag(a) W1 formed in fp32 and
// carried as two bf16 matrices so that the product keeps 16 significant bits of it; fp32 accumulation over
// all neurons, one rounding to bf16.  Uses the batched path's buffers as temporaries (they are filled later).
tardis_status_t launch_fold_tensor(Handle* H, const tardis_fold_desc_t* desc, cudaStream_t s) {
  State* S = static_cast<State*>(H->bstate);
  if (!S || H->dtype != TARDIS_BF16) return TARDIS_ERR_UNSUPPORTED;
  const int d = H->d, h = H->h;
  dim3 tb(32, 8);
  k_scale_transpose_split<<<dim3((d + 63) / 64, (h + 63) / 64), 256, 0, s>>>(static_cast<const uint32_t*>(H->W1), H->a, reinterpret_cast<uint32_t*>(S->What_hi),
                                                                             reinterpret_cast<uint32_t*>(S->What_lo), h, d);
  const size_t cap = size_t(kChunkCapture) * h;              // floats in the score buffer
  int rows_per = int(cap / d);
  rows_per = rows_per / 128 * 128;
  if (rows_per < 128) return TARDIS_ERR_UNSUPPORTED;
  for (int i0 = 0; i0 < d; i0 += rows_per) {
    const int rows = d - i0 < rows_per ? d - i0 : rows_per;
    GemmArgs g = {};
    g.M = rows; g.N = d; g.K1 = h; g.K2 = desc->flags == TARDIS_FOLD_BF16_INTERMEDIATE ? 0 : h;   // (study mode: leading term only)
    g.A1 = static_cast<const __nv_bfloat16*>(desc->W2) + size_t(i0) * h; g.lda1 = h; g.B1 = S->What_hi; g.ldb1 = h;
    g.A2 = g.A1; g.lda2 = h; g.B2 = S->What_lo; g.ldb2 = h;
    g.epilogue = GEMM_EPI_F32; g.out_f32 = S->zhat; g.ldo = d; g.error_word = &H->counters[CTR_ERROR];
    const tardis_status_t st = launch_gemm(g, s);
    if (st != TARDIS_OK) return st;
    k_store_folded<<<dim3((d + 31) / 32, (rows + 31) / 32), tb, 0, s>>>(S->zhat, static_cast<__nv_bfloat16*>(H->C), i0, rows, d);
  }
  TARDIS_CUDA_TRY(cudaGetLastError());
  return TARDIS_OK;
}

tardis_status_t batched_finish(Handle* H, const void* W2, cudaStream_t s) {
  State* S = static_cast<State*>(H->bstate);
  if (!S) return TARDIS_OK;
  const int d = H->d, h = H->h;
  const size_t hd = size_t(h) * d;
  // W_f[i][k] row-major (the GEMMs want the channel index contiguous in both operands): transpose of C
  TARDIS_CUDA_TRY(launch_transpose(static_cast<const __nv_bfloat16*>(H->C), S->Wf, d, d, s));
  if (W2) TARDIS_CUDA_TRY(cudaMemcpyAsync(S->W2, W2, hd * 2, cudaMemcpyDeviceToDevice, s));
  else      // (a handle read back from a file has only the transposed copy)
    TARDIS_CUDA_TRY(launch_transpose(static_cast<const __nv_bfloat16*>(H->W2T), S->W2, h, d, s));
  TARDIS_CUDA_TRY(cudaMemsetAsync(S->lo_used, 0, size_t((h + 127) / 128) * 4, s));
  if (H->bits <= 4)   // (8-bit codes: the batched path is not used, see the dispatch)
    k_dequant_split<<<h, 256, 0, s>>>(H->codes, static_cast<const __nv_bfloat16*>(H->scale), H->zero, S->What_hi, S->What_lo,
                                    S->smaxrow, S->lo_used, d, H->G, H->bits);
  TARDIS_CUDA_TRY(cudaGetLastError());
  return few_finish(H, S->W2, S->Wf, s);
}

void batched_release(Handle* H) {
  State* S = static_cast<State*>(H->bstate);
  if (!S) return;
  void* ptrs[] = {S->Wf, S->W2, S->What_hi, S->What_lo, S->smaxrow, S->lo_used, S->zhat, S->yacc, S->x1, S->delta, S->bitmap, S->rlist, S->rcount};
  for (void* q : ptrs)
    if (q) dev_free(q);
  delete S;
  H->bstate = nullptr;
}

tardis_status_t launch_batched_forward(Handle* H, const void* xv, void* yv, int64_t n_total, cudaStream_t s) {
  State* S = static_cast<State*>(H->bstate);
  if (!S) return TARDIS_ERR_UNSUPPORTED;
  const int d = H->d, h = H->h;
  if (H->few && n_total <= 128 && !H->deterministic) return launch_few_forward(H, xv, yv, int(n_total), S->smaxrow, s);
  const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(xv);
  __nv_bfloat16* y = static_cast<__nv_bfloat16*>(yv);
  const bool keep_scores = H->dbg_bitmap || H->dbg_scores;
  const int chunk = keep_scores ? kChunkCapture : kChunk;
  for (int64_t t0 = 0; t0 < n_total; t0 += chunk) {
    const int n = int(n_total - t0 < chunk ? n_total - t0 : chunk);
    const __nv_bfloat16* xc = x + size_t(t0) * d;
    TARDIS_CUDA_TRY(cudaMemsetAsync(S->rcount, 0, size_t(n) * 4, s));
    k_xnorm<<<n, 256, 0, s>>>(xc, d, S->x1);
    // 1. fast scores: one GEMM over the hi and lo halves of the dequantised predictor
    GemmArgs g = {};
    g.M = n; g.N = h; g.K1 = d; g.K2 = d;
    g.A1 = xc; g.lda1 = d; g.B1 = S->What_hi; g.ldb1 = d; g.A2 = xc; g.lda2 = d; g.B2 = S->What_lo; g.ldb2 = d; g.second_used = S->lo_used;
    // its epilogue turns the scores into flag words and queues the pairs too close to a range end; the scores
    // themselves are stored only for the debug capture
    g.epilogue = GEMM_EPI_FLAGS; g.out_f32 = keep_scores ? S->zhat : nullptr; g.ldo = h; g.bias = H->b1;
    g.error_word = &H->counters[CTR_ERROR];
    g.lo = H->lo; g.hi = H->hi; g.colscale = S->smaxrow; g.rowscale = S->x1; g.keps = kEps * float((1 << H->bits) - 1);
    g.bitmap_out = S->bitmap; g.rlist = S->rlist; g.rcount = S->rcount; g.rcap = max_recheck(h);
    g.bits = H->bits;
    tardis_status_t st = launch_gemm(g, s);
    if (st != TARDIS_OK) return st;
    const bool staged = d <= 24576;                        // (192 KB)
    const size_t room = staged ? size_t(d / 16 + 1) * 16 * sizeof(double) : 0;
    const auto recheck = H->bits == 2 ? (staged ? k_recheck<2, true> : k_recheck<2, false>)
                                      : (H->bits == 4 ? (staged ? k_recheck<4, true> : k_recheck<4, false>) : (staged ? k_recheck<0, true> : k_recheck<0, false>));
    if (room > 48 * 1024) TARDIS_CUDA_TRY(cudaFuncSetAttribute(recheck, cudaFuncAttributeMaxDynamicSharedMemorySize, int(room)));
    recheck<<<n, 256, room, s>>>(S->rlist, S->rcount, H->codes, static_cast<const __nv_bfloat16*>(H->scale), H->zero, H->b1, H->lo, H->hi, xc, d, h,
                                 H->G, H->bits, S->bitmap, keep_scores ? S->zhat : nullptr, H->counters);
    if (H->dbg_bitmap || H->dbg_scores) {
      const size_t cnt = size_t(n) * h;
      k_capture<<<unsigned((cnt + 255) / 256), 256, 0, s>>>(S->bitmap, S->zhat, S->x1, n, h,
                                                            H->dbg_bitmap ? H->dbg_bitmap + size_t(t0) * (h / 32) : nullptr,
                                                            H->dbg_scores ? H->dbg_scores + size_t(t0) * h : nullptr);
    }
    // 2. result fixing: exact pre-activations of every neuron, masked correction
    GemmArgs z = {};
    z.M = n; z.N = h; z.K1 = d; z.A1 = xc; z.lda1 = d; z.B1 = H->W1; z.ldb1 = d;
    z.epilogue = GEMM_EPI_DELTA; z.out_bf16 = S->delta; z.ldo = h; z.bias = H->b1; z.a = H->a; z.c = H->c; z.bitmap = S->bitmap;
    z.act = H->act; z.error_word = &H->counters[CTR_ERROR];
    st = launch_gemm(z, s);
    if (st != TARDIS_OK) return st;
    // 3. y = X W_f^T + b_f + Delta W2^T, one product over d + h channels (two products that meet in an fp32 array write and read it and
    // end in a partial wave of CTAs each: 16384 tokens of 4096 / 16384 6.64 ms, now 6.30).  A batch of one tile of tokens is bound by weight traffic and has few tiles: it splits its
    // channel range over several CTAs, which add into the fp32 accumulator.
    // (not in deterministic mode: the order of those additions is not fixed)
    const int splits = (n <= kSplitTokens && d <= 8192 && !H->deterministic) ? 4 : 1;
    GemmArgs o = {};
    o.M = n; o.N = d; o.K1 = d; o.A1 = xc; o.lda1 = d; o.B1 = S->Wf; o.ldb1 = d; o.K2 = h; o.A2 = S->delta; o.lda2 = h; o.B2 = S->W2; o.ldb2 = h;
    o.ldo = d; o.bias = H->bf; o.error_word = &H->counters[CTR_ERROR];
    if (splits > 1) {
      TARDIS_CUDA_TRY(cudaMemsetAsync(S->yacc, 0, size_t(n) * d * sizeof(float), s));
      o.epilogue = GEMM_EPI_F32; o.out_f32 = S->yacc; o.splits = splits;
    } else {
      o.epilogue = GEMM_EPI_BF16; o.out_bf16 = y + size_t(t0) * d;
    }
    st = launch_gemm(o, s);
    if (st != TARDIS_OK) return st;
    if (splits > 1) {
      const size_t cnt = size_t(n) * d;
      k_round_store<<<unsigned((cnt / 4 + 255) / 256 + 1), 256, 0, s>>>(S->yacc, y + size_t(t0) * d, cnt);
    }
    H->launches += 5 + (splits > 1 ? 1 : 0) + ((H->dbg_bitmap || H->dbg_scores) ? 1 : 0);
  }
  TARDIS_CUDA_TRY(cudaGetLastError());
  return TARDIS_OK;
}

}  // namespace tardis
