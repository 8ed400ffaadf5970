// The online path (Section 5.4) for calls of a few to 128 tokens on bf16 layers with 2-bit or 4-bit codes, sm_100a.
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
//   Both take part in the programmatic hand-over: a CTA of k_few_out fills its stages with W2, one of k_few_in its stages with W1, as
//     soon as the launch before has left its SM, while other SMs still finish that one (two CTAs do not fit on an SM: the rings
//     take 200 KB and more).
//   4-bit codes take the same way with two bf16 terms per weight: 4096 / 16384, caches cold, 95 us for one token and 130 for 64, where
//     the dense products over a dequantised predictor took 200 and 181.
#include <string.h>

#include <algorithm>
#include <new>

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
constexpr int BARS = 512;                 // bytes for barriers and a few words behind the stages
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

template <int N, int BITS> struct InCfg {
  static constexpr int X_BYTES = N * BK * 2, STAGE = W_BYTES + X_BYTES;
  static constexpr int NS = N == 128 ? 6 : (N == 64 ? 9 : (N == 32 ? 11 : 12));
  // expanded predictor blocks in TMEM (32 columns each).  4-bit codes come as two blocks each, and their expansion waits for the launch
  // before anyway: as many as fit (3328 / 13312, 40 tokens: 80 us with six, 95 with two); 2-bit codes are no faster with six
  static constexpr int NBUF = N == 128 ? 4 : (BITS == 4 ? 8 : (N == 64 ? 2 : 4));
  static constexpr int COL_S = 0, COL_Z = N, COL_F = 2 * N, COL_A = 3 * N;
  // (an allocation is a power of two; a kernel that takes all 512 columns does so only behind the wait, they may be another's until then)
  static constexpr int TMEM = COL_A + NBUF * 32 <= 256 ? 256 : 512;
  static constexpr int SMEM = 1024 + NS * STAGE + BARS + MAX_NEAR * 16 + BM * ((N + 31) / 32) * 4 + N * 8;
  static_assert((2 * NS + 2 * NBUF + 5) * 8 + 16 + 64 <= BARS, "barriers, parts of re-evaluated scores");
  static_assert(SMEM <= 232448, "shared memory");
};
template <int N> struct OutCfg {
  static constexpr int X_BYTES = N * BK * 2, STAGE = W_BYTES + X_BYTES;
  static constexpr int NS = N == 128 ? 6 : (N == 64 ? 9 : 10);
  static constexpr int TMEM = N < 32 ? 32 : N;
  static constexpr int SMEM = 1024 + NS * STAGE + BARS;
  static_assert((2 * NS + 2) * 8 + 16 <= BARS, "barriers");
  static_assert(SMEM <= 232448, "shared memory");
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
  const float s = __uint_as_float(meta & 0xffff0000u), zp = float(meta & 15u);
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

// The same with 4-bit codes, one field at a time into the low mantissa bits: s (q - zp) has up to 12 significant bits, so there are
// always two terms, the rounded product and what it leaves (both exact: one fused multiply-add).
template <int TERM> __device__ __forceinline__ void expand_4bit(const uint4 (&code)[2], uint32_t meta, uint32_t (&out)[32]) {
  const __nv_bfloat162 off = as_bf2(pair_of(128.f + float(meta & 15u))), s = as_bf2(pair_of(__uint_as_float(meta & 0xffff0000u)));
  const uint32_t words[8] = {code[0].x, code[0].y, code[0].z, code[0].w, code[1].x, code[1].y, code[1].z, code[1].w};
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const __nv_bfloat162 v = __hsub2(as_bf2(((words[k] >> (4 * p)) & 0x000f000fu) | 0x43004300u), off), hi = __hmul2(v, s);
      out[k * 4 + p] = as_u32(TERM == 0 ? hi : __hfma2(v, s, __hneg2(hi)));
    }
}

// Exact fp64 predictor sum of one neuron and token over the code words first, first + step, ..., from the packed blocks the CTA
// has just read (`rows` apart).  A lone warp waits for its loads and for its instructions, nothing else (8 us per pair with the
// words read one after the other): four words' loads go out before the first is used, and the code is kept short.
template <int BITS> __device__ __noinline__ double exact_from_packed(const uint4* __restrict__ codes, const uint32_t* __restrict__ meta, const __nv_bfloat16* __restrict__ x,
                                                 int nwords, int kpg, int rows, int first, int step) {
  constexpr int PER = 32 / BITS, VEC = BITS / 2;           // codes of a word, 16-byte vectors of a block's neuron
  constexpr uint32_t MASK = (1u << BITS) - 1u;
  double acc = 0.0;
#pragma unroll 1
  for (int w0 = first; w0 < nwords; w0 += 4 * step) {
    uint32_t code[4], m[4];
    uint4 xv[4][PER / 8];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int w = w0 + u * step;
      if (w < nwords) {
        code[u] = reinterpret_cast<const uint32_t*>(codes + size_t(w >> 2) * rows)[w & 3];
        m[u] = meta[size_t(w / (4 * VEC) / kpg) * rows];
#pragma unroll
        for (int q = 0; q < PER / 8; ++q) xv[u][q] = *reinterpret_cast<const uint4*>(x + w * PER + q * 8);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (w0 + u * step >= nwords) break;
      const float zp = float(m[u] & 15u);
      double p0 = 0.0, p1 = 0.0;
#pragma unroll
      for (int p = 0; p < PER / 2; ++p) {                  // (q - zp) x is exact in fp32
        const uint4& xq = xv[u][p >> 2];
        const uint32_t xw = (p & 3) == 0 ? xq.x : ((p & 3) == 1 ? xq.y : ((p & 3) == 2 ? xq.z : xq.w));
        p0 += double((float((code[u] >> (BITS * p)) & MASK) - zp) * __uint_as_float(xw << 16));
        p1 += double((float((code[u] >> (16 + BITS * p)) & MASK) - zp) * __uint_as_float(xw & 0xffff0000u));
      }
      acc += double(__uint_as_float(m[u] & 0xffff0000u)) * (p0 + p1);
    }
  }
  return acc;
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

// N: token columns (the call's tokens rounded up); TERMS: bf16 terms of a correction (2 keeps 16 significant bits of it); BITS: of a
// code
template <int N, int TERMS, int BITS>
__global__ void __launch_bounds__(NT_IN, 1)            // (one CTA per SM: its shared memory)
k_few_in(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmWf, const __grid_constant__ CUtensorMap tmX,
         const InParams p) {
  using C = InCfg<N, BITS>;
  constexpr int VEC = BITS / 2, AHEAD = BITS == 2 ? 4 : 2;   // 16-byte vectors of a block's neuron; blocks fetched ahead (in registers)
  constexpr int RING = C::NBUF / 2;                    // expanded blocks per group of four warps
  constexpr int HALF = N / 2;                          // token columns per epilogue thread
  constexpr int MW = (HALF + 31) / 32;                 // flag words of a thread
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::NS * C::STAGE);   // [NS] stage filled
  uint64_t* empty = full + C::NS;                      // [NS] stage read by the MMAs and the norms
  uint64_t* a_full = empty + C::NS;                    // [NBUF] predictor block expanded
  uint64_t* a_empty = a_full + C::NBUF;                // [NBUF] ... and read
  uint64_t* acc_full = a_empty + C::NBUF;              // scores and pre-activations of a tile complete
  uint64_t* acc_free = acc_full + 1;
  uint64_t* f_full = acc_free + 1;                     // a piece of the folded product complete
  uint64_t* f_free = f_full + 1;
  uint64_t* norm_ready = f_free + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(norm_ready + 1);
  volatile uint32_t* failed = tmem_slot + 1;
  uint32_t* near_count = tmem_slot + 2;
  double* near_part = reinterpret_cast<double*>(smem + C::NS * C::STAGE + BARS - 64);   // [8 warps]
  uint4* near = reinterpret_cast<uint4*>(smem + C::NS * C::STAGE + BARS);         // [MAX_NEAR] row << 8 | token, lo, hi, b1
  uint32_t* settled = reinterpret_cast<uint32_t*>(near + MAX_NEAR);               // [BM][(N + 31) / 32] re-evaluated scores that are outside
  float* x1 = reinterpret_cast<float*>(settled + BM * ((N + 31) / 32));           // [N] sum |x|
  unsigned int* tok_flagged = reinterpret_cast<unsigned int*>(x1 + N);            // [N]

  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp: uniform, and known to be)
  const int nkb = p.nkb;
  const int2 wf = p.wf_plan[blockIdx.x];
  pdl_launch();
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 3); }
    for (int b = 0; b < C::NBUF; ++b) { mbar_init(&a_full[b], 4); mbar_init(&a_empty[b], 1); }
    mbar_init(acc_full, 1); mbar_init(acc_free, 8); mbar_init(f_full, 1); mbar_init(f_free, 8); mbar_init(norm_ready, 2);
    *failed = 0u;
    *near_count = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < BM * ((N + 31) / 32); i += NT_IN) settled[i] = 0u;
  if (threadIdx.x < N) tok_flagged[threadIdx.x] = 0u;
  __syncthreads();
  // (warp 0 goes on with its copies meanwhile)
  if (warp == 1) {
    if (C::TMEM > 256) pdl_wait();
    tmem_alloc(tmem_slot, C::TMEM);
  }
  if (warp != 0) {
    tc_fence_before();
    asm volatile("bar.sync 2, 352;" ::: "memory");
    tc_fence_after();
  }
  const uint32_t tmem = *tmem_slot;
  // The waits below are bounded, so none of them may begin before the launch before this one has ended: it may take any time.
  int issued = 0;                                      // fills of a stage, by warp 0

  if (warp == 0) {
    // ---------------- TMA: W1 tiles, then the folded matrix's blocks; the tokens beside each ----------------
    Walk w(p, wf), first = w;
    const int ahead = min(C::NS, w.total);
    auto bytes = [&](const Walk& at) { return uint32_t((at.folded ? BM : p.rows) * BK * 2 + C::X_BYTES); };
    auto weights = [&](const Walk& at, int s) { tma_load_2d_once(smem + s * C::STAGE, at.folded ? &tmWf : &tmW1, at.kb * BK, at.row0, &full[s]); };
    auto tokens = [&](const Walk& at, int s) { tma_load_2d(smem + s * C::STAGE + W_BYTES, &tmX, at.kb * BK, 0, &full[s]); };
    for (int s = 0; s < ahead; ++s, w.next())              // constant state: before the wait
      if (elect_one()) { mbar_expect_tx(&full[s], bytes(w)); weights(w, s); }
    pdl_wait();
    for (int s = 0; s < ahead; ++s, first.next())
      if (elect_one()) tokens(first, s);
    issued = ahead;
    for (int s = 0, parity = 0; issued < w.total; ++issued, w.next()) {
      if (!mbar_wait_issue(&empty[s], parity, failed)) break;
      if (elect_one()) { mbar_expect_tx(&full[s], bytes(w)); weights(w, s); tokens(w, s); }
      if (++s == C::NS) { s = 0; parity ^= 1; }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    constexpr uint32_t idesc = instr_desc_bf16(BM, N);
    const uint64_t wdesc = smem_desc_k_major_sw128(smem_u32(smem)), xdesc = smem_desc_k_major_sw128(smem_u32(smem) + W_BYTES);
    int s = 0, parity = 0, ati = 0, own0 = 0, own1 = 0;    // stage and its phase; tiles; expanded blocks used of either group
    auto next_stage = [&]() { if (++s == C::NS) { s = 0; parity ^= 1; } };
    pdl_wait();
    for (int tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++ati) {
      const int terms = BITS > 2 || p.two_terms[tile] ? 2 : 1;
      bool ok = mbar_wait_issue(acc_free, (ati & 1) ^ 1, failed);
      for (int kb = 0; kb < nkb; ++kb) {
        ok = mbar_wait_issue(&full[s], parity, failed);
        tc_fence_after();
        const uint64_t da = wdesc + uint32_t(s * (C::STAGE >> 4)), db = xdesc + uint32_t(s * (C::STAGE >> 4));
        if (elect_one() && ok) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) umma_f16(tmem + C::COL_Z, da + k * 2, db + k * 2, idesc, (kb | k) != 0 ? 1u : 0u);
        }
        for (int term = 0; term < terms; ++term) {
          const int own = (kb & 1) ? own1 : own0, b = (kb & 1) + 2 * (own % RING);
          ok = mbar_wait_issue(&a_full[b], (own / RING) & 1, failed);
          tc_fence_after();
          if (elect_one() && ok) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_f16_ta(tmem + C::COL_S, tmem + C::COL_A + b * 32 + k * 8, db + k * 2, idesc, (kb | k | term) != 0 ? 1u : 0u);
            umma_commit(&a_empty[b]);
            if (term == terms - 1) umma_commit(&empty[s]);
          }
          if (kb & 1) ++own1; else ++own0;
        }
        next_stage();
      }
      if (elect_one() && ok) umma_commit(acc_full);
    }
    for (int u = wf.x, end = wf.x / nkb * nkb, seg = 0; u < wf.y; ++seg) {
      end = min(wf.y, end + nkb);                            // blocks of one output tile
      bool ok = mbar_wait_issue(f_free, (seg & 1) ^ 1, failed);
      for (uint32_t accumulate = 0u; u < end; ++u) {
        ok = mbar_wait_issue(&full[s], parity, failed);
        tc_fence_after();
        const uint64_t da = wdesc + uint32_t(s * (C::STAGE >> 4)), db = xdesc + uint32_t(s * (C::STAGE >> 4));
        if (elect_one() && ok) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) umma_f16(tmem + C::COL_F, da + k * 2, db + k * 2, idesc, k ? 1u : accumulate);
          umma_commit(&empty[s]);
        }
        accumulate = 1u;
        next_stage();
      }
      if (elect_one() && ok) umma_commit(f_full);
    }
  } else if (warp < 4) {
    // ---------------- token norms sum |x|, read beside the MMAs while the first tile passes by ----------------
    const int total = Walk(p, wf).total;
    const bool any_tile = int(blockIdx.x) < p.ntiles;
    // A stage goes back only when they have read it, so they must not take longer than the MMAs: LPT lanes per token, each with its
    // 16-byte pieces of a 128-byte row, four sums side by side (one lane per token and one chain of additions: 5 us per call).
    constexpr int LPT = N >= 64 ? 1 : 64 / N, TPL = N > 64 ? N / 64 : 1, PIECES = 8 / LPT;
    float sum[TPL][4] = {};
    const int me = (warp - 2) * 32 + lane;
    pdl_wait();
    for (int i = 0, s = 0, parity = 0; i < total; ++i) {
      if (!mbar_wait_warp(&full[s], parity)) { *failed = 1u; break; }
      if (any_tile && i < nkb) {
        const uint8_t* xt = smem + s * C::STAGE + W_BYTES;
#pragma unroll
        for (int r = 0; r < TPL; ++r) {
          const int t = me / LPT + 64 * r;
#pragma unroll
          for (int c = 0; c < PIECES; ++c) {
            const uint4 v = *reinterpret_cast<const uint4*>(xt + t * 128 + (((c * LPT + me % LPT) ^ (t & 7)) << 4));
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) sum[r][q] += fabsf(__uint_as_float(w[q] << 16)) + fabsf(__uint_as_float(w[q] & 0xffff0000u));
          }
        }
        if (i == nkb - 1) {
#pragma unroll
          for (int r = 0; r < TPL; ++r) {
            float tot = (sum[r][0] + sum[r][1]) + (sum[r][2] + sum[r][3]);   // (inf or NaN where the token holds one)
#pragma unroll
            for (int o = LPT / 2; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
            if (me % LPT == 0) x1[me / LPT + 64 * r] = tot <= 3.0e38f ? tot : __int_as_float(0x7f800000);
          }
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&empty[s]);
        if (i == nkb - 1) mbar_arrive(norm_ready);
      }
      if (++s == C::NS) { s = 0; parity ^= 1; }
    }
  } else {
    // ---------------- predictor expansion, then the epilogues: thread = weight row 32 q + lane of the tile ----------------
    const int q = warp & 3, gi = (warp - 4) >> 2;          // TMEM lanes 32 q .. + 31; channel blocks / token columns of this group
    const uint32_t lanes = tmem + (uint32_t(q * 32) << 16);
    const int row = q * 32 + lane, rows = p.rows;
    const bool holds = q * 32 < rows;                      // any row of this warp is in use
    const int kpg = p.G / BK;                              // channel blocks per predictor group
    int ati = 0, own = 0;
    bool ok = true;
    // (after a wait that ran out the flow stays the same, without further waits: the warps meet at named barriers)
    for (int tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++ati) {
      // -- this group's channel blocks gi, gi + 2, ...: codes fetched some blocks ahead --
      const int terms = BITS > 2 || p.two_terms[tile] ? 2 : 1;
      const uint4* const tile_codes = p.codes + size_t(tile) * nkb * VEC * rows;
      const uint32_t* const tile_meta = p.meta + size_t(tile) * (p.d / p.G) * rows;
      const int mine = (nkb - gi + 1) / 2;
      uint4 code[AHEAD][VEC] = {};
      uint32_t meta[AHEAD] = {};
      auto fetch = [&](int kb, uint4 (&cd)[VEC], uint32_t& mt) {
        if (row < rows) {
#pragma unroll
          for (int q = 0; q < VEC; ++q) cd[q] = __ldg(tile_codes + size_t(kb * VEC + q) * rows + row);
          mt = __ldg(tile_meta + size_t(kb / kpg) * rows + row);
        }
      };
#pragma unroll
      for (int u = 0; u < AHEAD; ++u)
        if (u < mine) fetch(gi + 2 * u, code[u], meta[u]);
      const int j = tile * rows + row;
      const bool real = row < rows && j < p.h;
      float lo = 0.f, hi = 0.f, b1 = 0.f, fa = 0.f, fc = 0.f;
      if (real) { lo = p.lo[j]; hi = p.hi[j]; b1 = p.b1[j]; fa = p.a[j]; fc = p.c[j]; }
      const float smax = real ? p.smax[j] : 0.f;
      if (terms == 2) pdl_wait();
      for (int i0 = 0; i0 < mine && ok; i0 += AHEAD) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
          const int i = i0 + u;
          if (i < mine && ok) {
            uint32_t w[32];
            for (int term = 0; term < terms && ok; ++term) {
              if (!holds) {}
              else if constexpr (BITS == 4) {
                if (term == 0) expand_4bit<0>(code[u], meta[u], w);
                else expand_4bit<1>(code[u], meta[u], w);
              }
              else if (terms == 1) expand<-1>(code[u][0], meta[u], w);
              else if (term == 0) expand<0>(code[u][0], meta[u], w);
              else expand<1>(code[u][0], meta[u], w);
              if (term == terms - 1 && i + AHEAD < mine) fetch(gi + 2 * (i + AHEAD), code[u], meta[u]);
              const int b = gi + 2 * (own % RING);
              if (u == RING && i0 == 0) pdl_wait();        // (a tile's first RING blocks of one term find their places free)
              ok = mbar_wait_warp(&a_empty[b], ((own / RING) & 1) ^ 1);
              if (!ok) { *failed = 1u; break; }
              tc_fence_after();
              if (holds) tmem_st32(lanes + C::COL_A + b * 32, w);
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&a_full[b]);
              ++own;
            }
          }
        }
      }
      pdl_wait();                                          // (from here on: data of earlier launches)
      // -- scores -> flags of this thread's neuron and token columns gi HALF .. + HALF - 1 --
      ok = ok && mbar_wait_warp(norm_ready, 0) && mbar_wait_warp(acc_full, ati & 1);
      if (!ok) *failed = 1u;
      tc_fence_after();
      // (loops over columns stay rolled: unrolled, their code outgrows the instruction cache and costs 20 us)
      uint64_t flags = 0, open = 0;                        // bit c: token column gi HALF + c; open: too close to a range end to tell
      // the terms of a score are at most (largest |q - zp|) smax |x| each: 3 only where a tile has such codes
      const float tau1 = (BITS > 2 ? 15.f : (terms == 2 ? 3.f : 2.f)) * kEps * smax;
      const int cols = real ? min(HALF, p.n - gi * HALF) : 0;   // (may be negative)
#pragma unroll 1
      for (int c0 = 0; c0 < HALF; c0 += 8) {
        float v[8];
        tmem_ld8(lanes + C::COL_S + gi * HALF + c0, v);
        uint32_t fl = 0u, op = 0u;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float xn = x1[gi * HALF + c0 + e], z = v[e] + b1, tau = fmaf(tau1, xn, 1e-30f);
          const bool finite = xn <= 3.0e38f;               // (a non-finite token: every neuron flagged)
          // (a token of zeros has no error, and its scores, the biases, may well lie on range ends)
          const bool near_end = finite && xn > 0.f && (fabsf(z - lo) <= tau || fabsf(z - hi) <= tau);
          fl |= uint32_t(!near_end && !(finite && lo <= z && z < hi)) << e;
          op |= uint32_t(near_end) << e;
          v[e] = finite ? z : __int_as_float(0x7fc00000);
        }
        const uint32_t valid = cols >= c0 + 8 ? 0xffu : (cols > c0 ? (1u << (cols - c0)) - 1u : 0u);
        flags |= uint64_t(fl & valid) << c0;
        open |= uint64_t(op & valid) << c0;
        if (p.dbg_scores)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (c0 + e < cols) p.dbg_scores[size_t(gi * HALF + c0 + e) * p.h + j] = double(v[e]);
      }
      for (uint64_t w = open; w; w &= w - 1) {             // rare
        const int t = gi * HALF + __ffsll((long long)w) - 1;
        const uint32_t slot = atomicAdd(near_count, 1u);
        if (slot < MAX_NEAR) near[slot] = make_uint4(uint32_t(row) << 8 | uint32_t(t), __float_as_uint(lo), __float_as_uint(hi), __float_as_uint(b1));
        else {                                             // list full: this thread settles the pair alone
          const double ze = exact_from_packed<BITS>(tile_codes + row, tile_meta + row, p.x + size_t(t) * p.d, nkb * 4 * VEC, kpg, rows, 0, 1) + double(b1);
          if (!(double(lo) <= ze && ze < double(hi))) flags |= 1ull << (t - gi * HALF);
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const uint32_t nn = *near_count;
      if (nn > 0) {                                        // (the same for all eight warps)
        // A warp per pair, eight at a time; of the last round's four or fewer the warps share out the channels: a round takes 4 to 6 us for a
        // whole row, two rounds of loads and of dependent sums, and the other warps would wait for it
        const uint32_t queued = min(nn, uint32_t(MAX_NEAR)), left = queued & 7u, alone = left <= 4 ? queued - left : queued;
        const uint32_t parts = left == 0 || left > 4 ? 1u : (left == 1 ? 8u : (left == 2 ? 4u : 2u));
        for (uint32_t e0 = 0; e0 < queued; e0 += 8) {
          const bool whole = e0 < alone;
          const uint32_t np = whole ? 1u : parts, e = e0 + uint32_t(warp - 4) / np, part = uint32_t(warp - 4) % np;
          if (e >= queued) break;
          const int r = int(near[e].x >> 8), t = int(near[e].x & 255u);
          double z = exact_from_packed<BITS>(tile_codes + r, tile_meta + r, p.x + size_t(t) * p.d, nkb * 4 * VEC, kpg, rows, int(part * 32) + lane, int(32 * np));
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
          if (lane != 0) continue;
          if (!whole) { near_part[warp - 4] = z; continue; }
          z += double(__uint_as_float(near[e].w));
          if (!(double(__uint_as_float(near[e].y)) <= z && z < double(__uint_as_float(near[e].z))))
            atomicOr(&settled[r * ((N + 31) / 32) + (t >> 5)], 1u << (t & 31));
          if (p.dbg_scores) p.dbg_scores[size_t(t) * p.h + tile * rows + r] = z;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        for (uint32_t e = alone; e < queued; ++e) {        // pairs in parts: settled by their neuron's thread
          const int r = int(near[e].x >> 8), t = int(near[e].x & 255u) - gi * HALF;
          if (r != row || t < 0 || t >= HALF) continue;
          double z = 0.0;
          for (uint32_t k = 0; k < parts; ++k) z += near_part[(e - alone) * parts + k];
          z += double(b1);
          if (!(double(lo) <= z && z < double(hi))) flags |= 1ull << t;
          if (p.dbg_scores) p.dbg_scores[size_t(gi * HALF + t) * p.h + j] = z;
        }
        if (threadIdx.x == 128) { atomicAdd(&p.counters[CTR_RECHECKS], (unsigned long long)nn); *near_count = 0u; }
        uint32_t* fix = &settled[row * ((N + 31) / 32)];
        if (HALF >= 32) {
#pragma unroll
          for (int m = 0; m < MW; ++m) { flags |= uint64_t(fix[gi * MW + m]) << (32 * m); fix[gi * MW + m] = 0u; }
        } else {
          flags |= (fix[0] >> (gi * HALF)) & ((1u << (HALF & 31)) - 1u);
        }
      }
      // -- counts per token; corrections act(z) - a z - c where flagged, zero elsewhere --
      // Evaluated for every element, without branches: a walk over the set bits alone waits for its lane with the most of them, and for one
      // activation after the other (64 columns of a tile: 5.9 us, now 3.1)
#pragma unroll 1
      for (int c0 = 0; c0 < HALF; c0 += 8) {
        const uint32_t bits = uint32_t(flags >> c0) & 0xffu;
        float v[8];
        tmem_ld8(lanes + C::COL_Z + gi * HALF + c0, v);
        uint32_t count = 0u;                               // lane e: flagged neurons of token column c0 + e
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint32_t word = __ballot_sync(0xffffffffu, (bits >> e) & 1u);
          if (lane == e) count = __popc(word);
          if (p.dbg_bitmap) {                              // (cleared before the launch; a tile may begin inside a word)
            const int t = gi * HALF + c0 + e;
            if (lane == 0 && t < p.n && word) {
              atomicOr(p.dbg_bitmap + size_t(t) * (p.h / 32) + (j >> 5), word << (j & 31));
              if ((j & 31) && (word >> (32 - (j & 31)))) atomicOr(p.dbg_bitmap + size_t(t) * (p.h / 32) + (j >> 5) + 1, word >> (32 - (j & 31)));
            }
          }
        }
        if (count && gi * HALF + c0 + lane < p.n) atomicAdd(&tok_flagged[gi * HALF + c0 + lane], count);
        if (p.act == TARDIS_ACT_GELU_TANH) {
#pragma unroll
          for (int e = 0; e < 8; ++e) { const float z = v[e] + b1; v[e] = gelu_tanh_f32(z) - fa * z - fc; }
        } else if (p.act == TARDIS_ACT_GELU_ERF) {
#pragma unroll
          for (int e = 0; e < 8; ++e) { const float z = v[e] + b1; v[e] = gelu_f32(z, TARDIS_ACT_GELU_ERF) - fa * z - fc; }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) { const float z = v[e] + b1; v[e] = gelu_f32(z, TARDIS_ACT_RELU) - fa * z - fc; }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (c0 + e < cols) {
            const int t = gi * HALF + c0 + e;
            const float dl = (bits >> e) & 1u ? v[e] : 0.f;
            const __nv_bfloat16 h0 = __float2bfloat16_rn(dl);
            p.delta[size_t(t) * p.h + j] = h0;
            if (TERMS == 2) p.delta[size_t(N + t) * p.h + j] = __float2bfloat16_rn(dl - __bfloat162float(h0));
          }
        }
      }
      if (HALF < 32) {                                     // (both groups' threads read the same word: cleared after both have)
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (gi == 0) settled[row] = 0u;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_free);
    }
    // -- pieces of the folded product: added to the fp32 accumulator --
    pdl_wait();
    int seg = 0;
    for (int u = wf.x; u < wf.y; ++seg) {
      const int m = u / nkb;
      u = min(wf.y, (m + 1) * nkb);
      ok = ok && mbar_wait_warp(f_full, seg & 1);
      if (!ok) { *failed = 1u; break; }
      tc_fence_after();
#pragma unroll 1
      for (int c0 = 0; c0 < HALF; c0 += 8) {
        float v[8];
        tmem_ld8(lanes + C::COL_F + gi * HALF + c0, v);
        add_outputs(p.yacc, p.d, p.n, gi * HALF + c0, m * BM + row, v);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(f_free);
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    const int t = threadIdx.x - 128;
    if (t < p.n && tok_flagged[t]) atomicAdd(&p.nfl[t], tok_flagged[t]);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *failed) atomicExch(&p.counters[CTR_ERROR], 1ull);
  if (warp == 0 && *failed) land_copies<C::NS>(full, issued);
  if (warp == 1) tmem_dealloc(tmem, C::TMEM);
}

// Corrections times W2.  N: columns (tokens rounded up, times the terms of a correction).  CTA c works on the pairs
// [c total / grid, (c + 1) total / grid) of (output tile, neuron block).
template <int N>
__global__ void __launch_bounds__(NT_OUT, 1)
k_few_out(const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmD, const OutParams p) {
  using C = OutCfg<N>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::NS * C::STAGE);
  uint64_t* empty = full + C::NS;
  uint64_t* acc_full = empty + C::NS;
  uint64_t* acc_free = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 1);
  volatile uint32_t* failed = tmem_slot + 1;
  uint32_t* last = tmem_slot + 2;
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp: uniform, and known to be)
  auto begin_of = [&](int c) { return int((long long)p.total * c / int(gridDim.x)); };
  const int begin = begin_of(blockIdx.x), end = begin_of(blockIdx.x + 1), nkb = p.nkb;
  int issued = 0;                                      // fills of a stage, by warp 0
  pdl_launch();
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(acc_full, 1);
    mbar_init(acc_free, 4);
    *failed = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp == 0) {
    int m = begin / nkb, kb = begin - m * nkb, xb = kb;      // next pair; neuron block of the next token tile
    auto weights = [&](int s) { tma_load_2d_once(smem + s * C::STAGE, &tmW2, kb * BK, m * BM, &full[s]); };
    auto corrections = [&](int s) { tma_load_2d(smem + s * C::STAGE + W_BYTES, &tmD, xb * BK, 0, &full[s]); };
    auto next_weights = [&]() { if (++kb == nkb) { kb = 0; ++m; } };
    auto next_corrections = [&]() { if (++xb == nkb) xb = 0; };
    const int total = end - begin, ahead = min(C::NS, total);
    for (int s = 0; s < ahead; ++s, next_weights())          // constant state: before the wait
      if (elect_one()) { mbar_expect_tx(&full[s], C::STAGE); weights(s); }
    pdl_wait();
    for (int s = 0; s < ahead; ++s, next_corrections())
      if (elect_one()) corrections(s);
    issued = ahead;
    for (int s = 0, parity = 0; issued < total; ++issued, next_weights(), next_corrections()) {
      if (!mbar_wait_issue(&empty[s], parity, failed)) break;
      if (elect_one()) { mbar_expect_tx(&full[s], C::STAGE); weights(s); corrections(s); }
      if (++s == C::NS) { s = 0; parity ^= 1; }
    }
  } else {
    // TMEM only once the launch before has given its own back (an allocation that has to wait blocks)
    pdl_wait();
    if (warp == 1) tmem_alloc(tmem_slot, C::TMEM);
    tc_fence_before();
    asm volatile("bar.sync 1, 160;" ::: "memory");      // (warps 1..5; warp 0 goes on with its copies)
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp == 1) {
      constexpr uint32_t idesc = instr_desc_bf16(BM, N);
      const uint64_t wdesc = smem_desc_k_major_sw128(smem_u32(smem)), xdesc = smem_desc_k_major_sw128(smem_u32(smem) + W_BYTES);
      int s = 0, parity = 0;
      for (int u = begin, stop = begin / nkb * nkb, seg = 0; u < end; ++seg) {
        stop = min(end, stop + nkb);                           // blocks of one output tile
        bool ok = mbar_wait_issue(acc_free, (seg & 1) ^ 1, failed);
        for (uint32_t accumulate = 0u; u < stop; ++u) {
          ok = mbar_wait_issue(&full[s], parity, failed);
          tc_fence_after();
          const uint64_t da = wdesc + uint32_t(s * (C::STAGE >> 4)), db = xdesc + uint32_t(s * (C::STAGE >> 4));
          if (elect_one() && ok) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) umma_f16(tmem, da + k * 2, db + k * 2, idesc, k ? 1u : accumulate);
            umma_commit(&empty[s]);
          }
          accumulate = 1u;
          if (++s == C::NS) { s = 0; parity ^= 1; }
        }
        if (elect_one() && ok) umma_commit(acc_full);
      }
    } else {
      const int q = warp & 3, row = q * 32 + lane, et = threadIdx.x - 64;
      const uint32_t lanes = tmem + (uint32_t(q * 32) << 16);
      if (blockIdx.x == 0) {                               // flagged neurons per token, counted by the launch before
        unsigned int f = et < p.n ? p.nfl[et] : 0u;
        if (et < p.n) p.nfl[et] = 0u;
        const unsigned int sum = __reduce_add_sync(0xffffffffu, f), most = __reduce_max_sync(0xffffffffu, f);
        if (lane == 0 && sum) {
          atomicAdd(&p.counters[CTR_FLAGGED_TOTAL], (unsigned long long)sum);
          atomicMax(&p.counters[CTR_FLAGGED_MAX], (unsigned long long)most);
        }
      }
      bool ok = true;
      int seg = 0;
      for (int u = begin; u < end; ++seg) {
        const int m = u / nkb, i = m * BM + row;
        u = min(end, (m + 1) * nkb);
        ok = ok && mbar_wait_warp(acc_full, seg & 1);
        if (!ok) *failed = 1u;
        tc_fence_after();
        const int cols = N / p.terms;                      // token columns; with two terms the second one is cols further on
#pragma unroll 1
        for (int c0 = 0; c0 < cols && c0 < p.n; c0 += 8) {
          float v[8];
          tmem_ld8(lanes + c0, v);
          if (p.terms == 2) {
            float w[8];
            tmem_ld8(lanes + cols + c0, w);
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] += w[e];
          }
          add_outputs(p.yacc, p.d, p.n, c0, i, v);
        }
        tc_fence_before();
        __threadfence();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_free);
        asm volatile("bar.sync 2, 128;" ::: "memory");
        if (et == 0) *last = atomicAdd(&p.done[m], 1u) + 1u == p.parts[m] ? 1u : 0u;
        asm volatile("bar.sync 2, 128;" ::: "memory");
        if (*last) {                                       // every part is in: b_f, one rounding; the accumulator is left cleared
          __threadfence();
          // (a lane takes four outputs, a warp every fourth token: its loads are in flight together)
          const int i4 = m * BM + lane * 4;
          if (i4 < p.d) {
            const float4 bf = *reinterpret_cast<const float4*>(p.bf + i4);
#pragma unroll 1
            for (int t0 = q; t0 < p.n; t0 += 16) {
              float4 v[4];
#pragma unroll
              for (int r = 0; r < 4; ++r)
                if (t0 + 4 * r < p.n) v[r] = __ldcg(reinterpret_cast<const float4*>(p.yacc + size_t(t0 + 4 * r) * p.d + i4));
#pragma unroll
              for (int r = 0; r < 4; ++r)
                if (t0 + 4 * r < p.n) {
                  const size_t at = size_t(t0 + 4 * r) * p.d + i4;
                  const __nv_bfloat162 o[2] = {__floats2bfloat162_rn(v[r].x + bf.x, v[r].y + bf.y), __floats2bfloat162_rn(v[r].z + bf.z, v[r].w + bf.w)};
                  *reinterpret_cast<uint2*>(p.y + at) = *reinterpret_cast<const uint2*>(o);
                  *reinterpret_cast<float4*>(p.yacc + at) = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
          }
          if (et == 0) p.done[m] = 0u;
        }
        asm volatile("bar.sync 2, 128;" ::: "memory");     // (*last has been read)
      }
    }
    tc_fence_before();
    asm volatile("bar.sync 1, 160;" ::: "memory");
    if (warp == 1) tmem_dealloc(tmem, C::TMEM);
  }
  __syncthreads();
  if (threadIdx.x == 0 && *failed) atomicExch(&p.counters[CTR_ERROR], 1ull);
  if (warp == 0 && *failed) land_copies<C::NS>(full, issued);
}

// ---- set-up ---------------------------------------------------------------------------------------------
// Packed predictor: block (tile of `rows` neurons, 64 channels) = rows x 16 bytes (4-bit codes: twice, 32 channels each), a neuron's
// four code words each with its even channels' codes in the lower half and the odd ones' in the upper half; per (tile, group)
// `rows` words, bf16 scale above, zero-point below.  two_terms (2-bit codes): the tile has a value with |q - zp| = 3.
template <int BITS>
__global__ void k_pack(const uint32_t* __restrict__ codes, const __nv_bfloat16* __restrict__ scale, const uint8_t* __restrict__ zero,
                       uint4* __restrict__ out, uint32_t* __restrict__ meta, uint32_t* __restrict__ two_terms, int rows, int d, int h, int G, int nkb) {
  constexpr int PER = 32 / BITS, VEC = BITS / 2;
  constexpr uint32_t MASK = (1u << BITS) - 1u;
  const int tile = blockIdx.x, r = threadIdx.x, j = tile * rows + r, ng = d / G;
  bool two = false;
  for (int v = blockIdx.y; v < nkb * VEC; v += gridDim.y) {
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (j < h) {
      const uint4 src = *reinterpret_cast<const uint4*>(codes + size_t(j) * (d / PER) + v * 4);
      const uint32_t s[4] = {src.x, src.y, src.z, src.w};
      const uint32_t zp = zero[size_t(j) * ng + v / VEC * BK / G] & MASK;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int p = 0; p < PER / 2; ++p)
          w[k] |= ((s[k] >> (2 * BITS * p)) & MASK) << (BITS * p) | ((s[k] >> (2 * BITS * p + BITS)) & MASK) << (16 + BITS * p);
        if (BITS == 2) {
          const uint32_t lo = s[k] & 0x55555555u, hi = (s[k] >> 1) & 0x55555555u;   // bits of the codes
          two |= (zp == 0u && (lo & hi)) || (zp == 3u && (~(lo | hi) & 0x55555555u));
        }
      }
    }
    out[(size_t(tile) * nkb * VEC + v) * rows + r] = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if (two) two_terms[tile] = 1u;
  for (int g = blockIdx.y; g < ng; g += gridDim.y)
    meta[(size_t(tile) * ng + g) * rows + r] =
        j < h ? (uint32_t(__bfloat16_as_ushort(scale[size_t(j) * ng + g])) << 16) | (zero[size_t(j) * ng + g] & MASK) : 0u;
}

// The shares of the folded product (end of each CTA's) and, per output tile, how many CTAs of k_few_out contribute to it (those that
// hold its first to its last pair), put where the kernels read them.
constexpr int MAX_GRID = 256;
struct Shares { int end[MAX_GRID]; };
__global__ void k_plan(const Shares shares, int2* plan, int grid, unsigned int* parts, int mtiles, int nkb, int out_grid) {
  for (int c = threadIdx.x; c < grid; c += blockDim.x) plan[c] = make_int2(c ? shares.end[c - 1] : 0, shares.end[c]);
  const long long total = (long long)mtiles * nkb;
  auto owner = [&](long long pair) {                       // the CTA c with total c / out_grid <= pair < total (c + 1) / out_grid
    int c = int(pair * out_grid / total);
    while (total * (c + 1) / out_grid <= pair) ++c;
    while (total * c / out_grid > pair) --c;
    return c;
  };
  for (int m = threadIdx.x; m < mtiles; m += blockDim.x)
    parts[m] = unsigned(owner((long long)(m + 1) * nkb - 1) - owner((long long)m * nkb) + 1);
}

struct State {
  uint4* codes; uint32_t *meta, *two_terms; int2* plan; float* yacc; unsigned int *nfl, *done, *parts;
  __nv_bfloat16* delta;
  CUtensorMap w1, w2, wf;
  int grid, out_grid, nkb, rows, ntiles, mtiles, out_nkb;
};

// Shares of the folded product's blocks: a neuron tile's block costs its rows' share of a 128-row one plus a seventh (codes);
// every CTA is filled up to the same total, and pieces of fewer than 8 blocks are not dealt (a piece costs one pass over a
// 128-row accumulator at its end).
static void deal_folded_blocks(const State& S, Shares& plan) {
  const double per_tile = 1.15 * S.rows / BM * S.nkb;
  const int blocks = S.mtiles * S.nkb;
  double room[MAX_GRID];
  auto fill = [&](double level) {
    double sum = 0.0;
    for (int c = 0; c < S.grid; ++c) {
      room[c] = level - per_tile * ((S.ntiles - c + S.grid - 1) / S.grid);
      if (room[c] < 8.0) room[c] = 0.0;
      sum += room[c];
    }
    return sum;
  };
  double lo = 0.0, hi = per_tile * (S.ntiles / S.grid + 2) + blocks + 8.0;      // (one CTA alone could take all)
  while (hi - lo > 1e-3) { const double mid = 0.5 * (lo + hi); (fill(mid) >= blocks ? hi : lo) = mid; }   // the level that holds all blocks
  const double sum = fill(hi);
  double cum = 0.0;
  for (int c = 0; c < S.grid; ++c) {
    cum += room[c];
    plan.end[c] = c == S.grid - 1 ? blocks : std::min(blocks, int(cum / sum * blocks + 0.5));
  }
}

}  // namespace few

using namespace few;

namespace {
// Serves bf16 layers with 2-bit or 4-bit codes in groups of a multiple of 64 channels (every channel block lies in one group).
bool served(const Handle* H) { return H->dtype == TARDIS_BF16 && (H->bits == 2 || H->bits == 4) && H->G % BK == 0 && tensor_maps_available(); }

State shape(const Handle* H) {
  State S = {};
  const int d = H->d, h = H->h;
  S.grid = std::min(H->num_sms, MAX_GRID);
  const int rounds = (h + S.grid * BM - 1) / (S.grid * BM), share = (h + S.grid * rounds - 1) / (S.grid * rounds);
  S.rows = std::min(BM, std::max(16, (share + 7) / 8 * 8));           // every CTA gets the same number of tiles, or one less
  S.nkb = d / BK; S.ntiles = (h + S.rows - 1) / S.rows; S.mtiles = (d + BM - 1) / BM; S.out_nkb = (h + BK - 1) / BK;
  return S;
}
struct Req { void** p; size_t bytes; };
struct Requests { Req r[6]; };                             // codes and meta, then scratch
Requests requests(const Handle* H, State* S) {
  return {{{reinterpret_cast<void**>(&S->codes), size_t(S->ntiles) * S->nkb * S->rows * 8 * H->bits},
           {reinterpret_cast<void**>(&S->meta), size_t(S->ntiles) * (H->d / H->G) * S->rows * 4},
           {reinterpret_cast<void**>(&S->plan), sizeof(int2) * S->grid}, {reinterpret_cast<void**>(&S->yacc), sizeof(float) * MAX_TOKENS * H->d},
           {reinterpret_cast<void**>(&S->nfl), sizeof(unsigned int) * (MAX_TOKENS + 2 * S->mtiles + S->ntiles)},
           {reinterpret_cast<void**>(&S->delta), size_t(2) * MAX_TOKENS * H->h}}};
}
}  // namespace

size_t few_room(const Handle* H) {
  if (!served(H)) return 0;
  State S = shape(H);
  size_t room = 0;
  for (const Req& r : requests(H, &S).r) room += dev_room(r.bytes);
  return room;
}

tardis_status_t few_prepare(Handle* H) {
  H->few = nullptr;
  if (!served(H)) return TARDIS_OK;
  State* S = new (std::nothrow) State(shape(H));
  if (!S) return TARDIS_ERR_ALLOC;
  H->few = S;
  const Requests all = requests(H, S);
  const Req (&reqs)[6] = all.r;
  for (const Req& r : reqs) {
    const cudaError_t e = dev_malloc(r.p, r.bytes);
    if (e != cudaSuccess) { set_last_error(e, "cudaMalloc"); cudaGetLastError(); few_release(H); return TARDIS_ERR_ALLOC; }
  }
  auto room = [](auto kernel, int smem) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); };
  const cudaError_t es[] = {room(k_few_in<16, 2, 2>, InCfg<16, 2>::SMEM), room(k_few_in<32, 1, 2>, InCfg<32, 2>::SMEM), room(k_few_in<64, 1, 2>, InCfg<64, 2>::SMEM),
                            room(k_few_in<128, 1, 2>, InCfg<128, 2>::SMEM), room(k_few_in<16, 2, 4>, InCfg<16, 4>::SMEM), room(k_few_in<32, 1, 4>, InCfg<32, 4>::SMEM),
                            room(k_few_in<64, 1, 4>, InCfg<64, 4>::SMEM), room(k_few_in<128, 1, 4>, InCfg<128, 4>::SMEM), room(k_few_out<32>, OutCfg<32>::SMEM),
                            room(k_few_out<64>, OutCfg<64>::SMEM), room(k_few_out<128>, OutCfg<128>::SMEM)};
  for (cudaError_t e : es)
    if (e != cudaSuccess) { set_last_error(e, "cudaFuncSetAttribute"); few_release(H); return TARDIS_ERR_CUDA; }
  S->done = S->nfl + MAX_TOKENS;
  S->parts = S->done + S->mtiles;
  S->two_terms = S->parts + S->mtiles;
  H->bytes_predictor += reqs[0].bytes + reqs[1].bytes;
  for (int i = 2; i < 6; ++i) H->bytes_scratch += reqs[i].bytes;
  return TARDIS_OK;
}

tardis_status_t few_finish(Handle* H, const void* W2, const void* Wf, cudaStream_t s) {
  State* S = static_cast<State*>(H->few);
  if (!S) return TARDIS_OK;
  const int d = H->d, h = H->h;
  if (!make_map(&S->w1, H->W1, h, d, d, S->rows) || !make_map(&S->w2, W2, d, h, h, BM) || !make_map(&S->wf, Wf, d, d, d, BM)) {
    few_release(H);                                    // (not served: the other kernels take these calls)
    return TARDIS_OK;
  }
  Shares shares;
  deal_folded_blocks(*S, shares);
  S->out_grid = std::max(1, std::min(S->grid, S->mtiles * S->out_nkb / 4));
  TARDIS_CUDA_TRY(cudaMemsetAsync(S->nfl, 0, sizeof(unsigned int) * (MAX_TOKENS + 2 * S->mtiles + S->ntiles), s));
  k_plan<<<1, 256, 0, s>>>(shares, S->plan, S->grid, S->parts, S->mtiles, S->out_nkb, S->out_grid);
  TARDIS_CUDA_TRY(cudaMemsetAsync(S->yacc, 0, sizeof(float) * MAX_TOKENS * d, s));
  auto pack = H->bits == 2 ? k_pack<2> : k_pack<4>;
  pack<<<dim3(S->ntiles, 8), S->rows, 0, s>>>(H->codes, static_cast<const __nv_bfloat16*>(H->scale), H->zero, S->codes, S->meta, S->two_terms,
                                              S->rows, d, h, H->G, S->nkb);
  TARDIS_CUDA_TRY(cudaGetLastError());
  return TARDIS_OK;
}

void few_release(Handle* H) {
  State* S = static_cast<State*>(H->few);
  if (!S) return;
  void* ptrs[] = {S->codes, S->meta, S->plan, S->yacc, S->nfl, S->delta};
  for (void* q : ptrs)
    if (q) dev_free(q);
  delete S;
  H->few = nullptr;
}

template <typename K, typename... Args>
static cudaError_t launch_overlapped(K kernel, int grid, int threads, size_t smem, cudaStream_t s, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int N, int TERMS>
static tardis_status_t launch_n(Handle* H, const __nv_bfloat16* x, __nv_bfloat16* y, int n, const float* smaxrow, cudaStream_t s) {
  State* S = static_cast<State*>(H->few);
  CUtensorMap tmx, tmd;
  if (!make_map(&tmx, x, n, H->d, H->d, N) || !make_map(&tmd, S->delta, MAX_TOKENS, H->h, H->h, N * TERMS)) return TARDIS_ERR_UNSUPPORTED;
  InParams a = {};
  a.n = n; a.d = H->d; a.h = H->h; a.G = H->G; a.nkb = S->nkb; a.ntiles = S->ntiles; a.rows = S->rows; a.act = H->act;
  a.codes = S->codes; a.meta = S->meta; a.two_terms = S->two_terms;
  a.lo = H->lo; a.hi = H->hi; a.a = H->a; a.c = H->c; a.b1 = H->b1; a.smax = smaxrow; a.x = x;
  a.wf_plan = S->plan; a.delta = S->delta; a.yacc = S->yacc; a.nfl = S->nfl; a.counters = H->counters;
  a.dbg_bitmap = H->dbg_bitmap; a.dbg_scores = H->dbg_scores;
  if (H->dbg_bitmap) TARDIS_CUDA_TRY(cudaMemsetAsync(H->dbg_bitmap, 0, size_t(n) * (H->h / 32) * 4, s));
  static_assert(InCfg<N, 2>::SMEM == InCfg<N, 4>::SMEM, "one size");
  TARDIS_CUDA_TRY(launch_overlapped(H->bits == 2 ? k_few_in<N, TERMS, 2> : k_few_in<N, TERMS, 4>, S->grid, NT_IN, InCfg<N, 2>::SMEM, s, S->w1, S->wf, tmx, a));
  OutParams o = {};
  o.n = n; o.d = H->d; o.h = H->h; o.nkb = S->out_nkb; o.total = S->mtiles * S->out_nkb; o.terms = TERMS;
  o.bf = H->bf; o.yacc = S->yacc; o.y = y; o.done = S->done; o.parts = S->parts; o.nfl = S->nfl; o.counters = H->counters;
  TARDIS_CUDA_TRY(launch_overlapped(k_few_out<N * TERMS>, S->out_grid, NT_OUT, OutCfg<N * TERMS>::SMEM, s, S->w2, tmd, o));
  H->launches += 2;
  return TARDIS_OK;
}

// 1 .. 128 tokens.  Corrections keep two bf16 terms up to 16 tokens, as on the fused path that serves smaller calls.
tardis_status_t launch_few_forward(Handle* H, const void* xv, void* yv, int n, const float* smaxrow, cudaStream_t s) {
  const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(xv);
  __nv_bfloat16* y = static_cast<__nv_bfloat16*>(yv);
  if (n <= 16) return launch_n<16, 2>(H, x, y, n, smaxrow, s);
  if (n <= 32) return launch_n<32, 1>(H, x, y, n, smaxrow, s);
  if (n <= 64) return launch_n<64, 1>(H, x, y, n, smaxrow, s);
  return launch_n<128, 1>(H, x, y, n, smaxrow, s);
}

}  // namespace tardis
