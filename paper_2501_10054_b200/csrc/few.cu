// The online path (Section 5.4) for calls of a few to 128 tokens on bf16 layers with 2-bit codes, sm_100a.
//
// With that many tokens nearly every neuron is flagged by some token, so all of W1, W2, W_f and the predictor has to be read,
// once: the bound is HBM (4096 / 16384: 320 MB = 49 us).  Two launches do the whole call; weights are the 128-row A operand
// of tcgen05.mma and the tokens its N columns, so a weight tile is read by exactly one CTA.
//
//   k_few_in: a CTA takes tiles of up to 128 neurons, of a size that gives every CTA the same share (4096 / 16384: 112 neurons,
//     147 tiles for 148 CTAs; with 128 neurons 20 CTAs had none).  One pass over the channels computes both the predictor
//     scores and the exact pre-activations of the tile, from the same token tile in shared memory: W1 arrives by TMA, the
//     predictor by plain loads of its packed codes (19 MB instead of the 134 MB of a dequantised matrix), expanded in registers
//     to the bf16 values s (q - zp) and written to TMEM, from where tcgen05.mma takes its A operand.  Scores -> flags (the ones
//     near a range end re-evaluated in fp64), pre-activations -> corrections (bf16) in global memory.  The folded product
//     X W_f^T needs only the tokens; its channel blocks are dealt to the CTAs so that all of them have about the same to do.
//   k_few_out: the corrections times W2, the (output tile, neuron block) pairs dealt evenly to the CTAs; partial outputs are
//     added to the fp32 accumulator, and the last CTA to contribute to an output tile rounds it to y and clears it.
//   Both take part in the programmatic hand-over: k_few_out fills its stages with W2 while k_few_in finishes, k_few_in its
//     stages with W1 while the launch before it finishes (both fit on an SM side by side up to 64 tokens).
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "common.cuh"
#include "tc.cuh"

namespace tardis {
namespace few {
using namespace tc;

constexpr int BM = 128;                   // weight rows per MMA tile
constexpr int BK = 64;                    // channels per stage
constexpr int W_BYTES = BM * BK * 2;
constexpr int NT_IN = 384;                // warp 0 TMA, 1 MMA, 2..3 token norms, 4..11 predictor expansion and epilogues
constexpr int NT_OUT = 192;               // warp 0 TMA, 1 MMA, 2..5 epilogue
constexpr int MAX_TOKENS = 128;
constexpr int MAX_NEAR = 256;             // scores near a range end per tile that can queue (further ones are settled in place)
constexpr float kEps = 7.62939453125e-6f; // 2^-17: accumulation-error allowance of the fast scores, relative to 3 max s |x|_1

struct InParams {
  int n, d, h, G, nkb, ntiles, rows, act; // nkb: channel blocks of 64; rows: neurons per tile (at most BM)
  const uint4* codes; const uint32_t* meta;       // packed predictor (see k_pack)
  const uint32_t* two_terms;              // per tile: some s (q - zp) need a second bf16 term
  const float *lo, *hi, *a, *c, *b1, *smax;
  const __nv_bfloat16* x;
  const int2* wf_plan;                    // per CTA: its blocks of the folded product, in (output tile, channel block) order
  __nv_bfloat16* delta;                   // [terms * N][h]
  float* yacc;                            // [N][d]
  unsigned int* nfl;                      // [MAX_TOKENS] flagged neurons per token
  unsigned long long* counters;
  uint32_t* dbg_bitmap; double* dbg_scores;
};
struct OutParams {
  int n, d, h, nkb, total, terms;         // nkb: neuron blocks of 64; total: (output tile, neuron block) pairs
  const float* bf; float* yacc; __nv_bfloat16* y;
  unsigned int* done; const unsigned int* parts;   // [output tiles] contributions so far, and how many there will be
  unsigned int* nfl; unsigned long long* counters;
};

template <int N> struct InCfg {
  static constexpr int X_BYTES = N * BK * 2, STAGE = W_BYTES + X_BYTES;
  static constexpr int NS = N == 128 ? 5 : (N == 64 ? 4 : (N == 32 ? 5 : 6));
  static constexpr int NBUF = 4;                                    // expanded predictor blocks in TMEM (32 columns each)
  static constexpr int COL_S = 0, COL_Z = N, COL_F = 2 * N, COL_A = 3 * N;
  static constexpr int TMEM = COL_A + NBUF * 32 <= 256 ? 256 : 512;
  static constexpr int SMEM = 1024 + NS * STAGE + 256 + MAX_NEAR * 16 + BM * ((N + 31) / 32) * 4 + N * 8 + 8 * 1024;
};
template <int N> struct OutCfg {
  static constexpr int X_BYTES = N * BK * 2, STAGE = W_BYTES + X_BYTES;
  static constexpr int NS = N == 128 ? 4 : (N == 64 ? 4 : 5);
  static constexpr int TMEM = N < 32 ? 32 : N;
  static constexpr int SMEM = 1024 + NS * STAGE + 256;
};

__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ uint32_t as_u32(__nv_bfloat162 v) { return *reinterpret_cast<uint32_t*>(&v); }
__device__ __forceinline__ __nv_bfloat162 as_bf2(uint32_t v) { return *reinterpret_cast<__nv_bfloat162*>(&v); }
__device__ __forceinline__ uint32_t pair_of(float v) { return as_u32(__float2bfloat162_rn(v)); }

// The 64 channels of one neuron expanded to bf16 pairs s (q - zp).  A code word holds the even channel of pair p in bits
// 2p, 2p + 1 and the odd one 16 bits above.  Three pairs at a time are masked where they are into the mantissa of 128.0 (which
// weights them by 1, 4 and 16), the offset (128 + weight zp) is subtracted and the scale over the weight multiplied: every step
// is exact in bf16 when |q - zp| <= 2.  TERM 0 / 1: the two terms of values with |q - zp| = 3 (clamped to 2, and the rest).
template <int TERM> __device__ __forceinline__ void expand(const uint4& code, uint32_t meta, uint32_t (&out)[32]) {
  const float s = __uint_as_float(meta & 0xffff0000u), zp = float(meta & 3u);
  const uint32_t words[4] = {code.x, code.y, code.z, code.w};
  __nv_bfloat162 off[3], sc[3], lim[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float w = float(1 << (2 * i));
    off[i] = as_bf2(pair_of(128.f + w * zp));
    sc[i] = as_bf2(pair_of(s / w));
    lim[i] = as_bf2(pair_of(2.f * w));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const int i = p % 3;
      const uint32_t m = ((words[k] >> (6 * (p / 3))) & (0x00030003u << (2 * i))) | 0x43004300u;
      __nv_bfloat162 v = __hsub2(as_bf2(m), off[i]);
      if (TERM >= 0) {
        const __nv_bfloat162 c = __hmin2(__hmax2(v, __hneg2(lim[i])), lim[i]);
        v = TERM == 0 ? c : __hsub2(v, c);
      }
      out[k * 8 + p] = as_u32(__hmul2(v, sc[i]));
    }
}

// Exact fp64 predictor sum of one neuron and token over the channel blocks first, first + step, ..., from the packed blocks the
// CTA has just read (`rows` apart).  A lone warp waits for its loads and its chains of additions, nothing else (8 us per pair
// with the words read one after the other): the loads of a block go out before the first is used, and four sums run side by side.
__device__ __noinline__ double exact_from_packed(const uint4* __restrict__ codes, const uint32_t* __restrict__ meta, const __nv_bfloat16* __restrict__ x,
                                                 int nkb, int kpg, int rows, int first, int step) {
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int kb = first; kb < nkb; kb += step) {
    const uint4 code = codes[size_t(kb) * rows];
    const uint32_t m = meta[size_t(kb / kpg) * rows];
    uint4 xv[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) xv[c] = *reinterpret_cast<const uint4*>(x + kb * BK + c * 8);
    const float zp = float(m & 3u);
    const uint32_t words[4] = {code.x, code.y, code.z, code.w};
    double part[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint4& q = xv[2 * k + (p >> 2)];
        const uint32_t xw = (p & 3) == 0 ? q.x : ((p & 3) == 1 ? q.y : ((p & 3) == 2 ? q.z : q.w));
        // (q - zp) x is exact in fp32
        part[k] += double((float((words[k] >> (2 * p)) & 3u) - zp) * __uint_as_float(xw << 16));
        part[k] += double((float((words[k] >> (16 + 2 * p)) & 3u) - zp) * __uint_as_float(xw & 0xffff0000u));
      }
    const double s = double(__uint_as_float(m & 0xffff0000u));
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] += s * part[k];
  }
  return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// Adds v[e], the value of output i (this lane's; outputs of a warp's lanes are consecutive, i of lane 0 a multiple of 4) for token
// t0 + e, to yacc.  Four lanes exchange values first, so that a lane adds four outputs of one token with one 128-bit reduction.
__device__ __forceinline__ void add_outputs(float* yacc, int d, int n, int t0, int i, const float (&v)[8]) {
  const int r = threadIdx.x & 3;
#pragma unroll
  for (int h = 0; h < 8; h += 4) {
    const float s0 = __shfl_xor_sync(0xffffffffu, (r & 1) ? v[h] : v[h + 1], 1);
    const float s1 = __shfl_xor_sync(0xffffffffu, (r & 1) ? v[h + 2] : v[h + 3], 1);
    // two outputs (this lane's pair) of tokens h + (r & 1) and h + 2 + (r & 1)
    const float a0 = (r & 1) ? s0 : v[h], a1 = (r & 1) ? v[h + 1] : s0, b0 = (r & 1) ? s1 : v[h + 2], b1 = (r & 1) ? v[h + 3] : s1;
    const float u0 = __shfl_xor_sync(0xffffffffu, (r & 2) ? a0 : b0, 2), u1 = __shfl_xor_sync(0xffffffffu, (r & 2) ? a1 : b1, 2);
    const int t = t0 + h + r;
    if (t < n && i < d) {
      float* const at = yacc + size_t(t) * d + (i & ~3);
      const float w0 = (r & 2) ? u0 : a0, w1 = (r & 2) ? u1 : a1, w2 = (r & 2) ? b0 : u0, w3 = (r & 2) ? b1 : u1;
      asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(at), "f"(w0), "f"(w1), "f"(w2), "f"(w3) : "memory");
    }
  }
}

// The sequence of a CTA's blocks: its neuron tiles, nkb blocks each, then its share of the folded product.  Stepped without
// divisions: one thread issues all copies (another all MMAs), and a step has to take less than the 300 ns in which a block
// arrives.
struct Walk {
  int nkb, ntiles, rows, step, tile, left, kb, row0, total;
  int2 wf;
  bool folded;
  __device__ __forceinline__ Walk(const InParams& p, int2 plan)
      : nkb(p.nkb), ntiles(p.ntiles), rows(p.rows), step(gridDim.x), tile(blockIdx.x), wf(plan), folded(false) {
    total = wf.y - wf.x;
    for (int t = tile; t < ntiles; t += step) total += nkb;
    begin_tile();
  }
  __device__ __forceinline__ void begin_tile() {
    if (tile < ntiles) { left = nkb; kb = 0; row0 = tile * rows; }
    else { folded = true; row0 = wf.x / nkb * BM; kb = wf.x % nkb; }
  }
  __device__ __forceinline__ void next() {
    if (++kb == nkb) { kb = 0; if (folded) row0 += BM; }
    if (!folded && --left == 0) { tile += step; begin_tile(); }
  }
};

