// bf16 GEMM on the 5th-generation tensor cores (see gemm.cuh for what it computes).
//
// A CTA computes 128 x BN tiles of the output, one after the other (persistent, one CTA per SM).  Warp 0 stages
// 128 x 64 (A) and BN x 64 (B) operand boxes into a ring of shared-memory stages with TMA
// (cp.async.bulk.tensor, 128-byte swizzle, no multicast); warp 1 issues tcgen05.mma (M = 128, N = BN,
// K = 16 per instruction; one elected lane), accumulating in tensor memory (TMEM, 128 lanes x BN fp32 columns,
// two accumulators used in turn) and releasing each stage with tcgen05.commit; warps 2..9 read a finished
// accumulator back with tcgen05.ld (each warp its own 32 lanes) and run the epilogue while the next tile's
// main loop fills the other accumulator.  Every wait on an mbarrier is bounded: when it runs out the waiter
// sets an error word and the CTA falls through to the end, where TMEM is released.
#include "gemm.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdio.h>

#include "common.cuh"
#include "tc.cuh"

namespace tardis {
namespace tc {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static const EncodeTiledFn fn = [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) != cudaSuccess) { cudaGetLastError(); return EncodeTiledFn(nullptr); }
    return q == cudaDriverEntryPointSuccess ? reinterpret_cast<EncodeTiledFn>(ptr) : EncodeTiledFn(nullptr);
  }();
  return fn;
}

bool tensor_maps_available() { return encode_fn() != nullptr; }

bool make_map(CUtensorMap* map, const void* base, int rows, int K, int ld, int box_rows) {
  const cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
  const cuuint64_t strides[1] = {cuuint64_t(ld) * 2};
  const cuuint32_t box[2] = {64, cuuint32_t(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  return encode_fn() && encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc

namespace gemm {
using namespace tc;

constexpr int BM = 128;                 // tile rows (tokens / outputs)
constexpr int BK = 64;                  // channels per stage: 64 bf16 = one 128-byte swizzle row
constexpr int NTHREADS = 320;           // warp 0 TMA, warp 1 MMA, warps 2..9 epilogue

struct KParams {
  int M, N, kb1, kb2;          // k blocks (of 64) of the two operand pairs
  const uint32_t* second_used; // per 128 rows n: bit 0 = the second pair adds something (null: it always counts), bit 1 = see fill_table
  int epilogue, ldo, act, splits;
  int fast_m, band;            // tile raster (see decode() in the kernel)
  float* out_f32; __nv_bfloat16* out_bf16;
  const float *bias, *a, *c;
  const uint32_t* bitmap;
  unsigned long long* error_word;
  const float *lo, *hi, *colscale, *rowscale;
  float keps;
  uint32_t* bitmap_out;
  uint32_t* rlist; unsigned int* rcount; int rcap, bits;
};

// CTAS: 1, or 2 for a pair of CTAs that works on 256 x BN tiles
template <int BN, int CTAS> struct Cfg {
  static constexpr int STAGE_BYTES = BM * BK * 2 + BN / CTAS * BK * 2;   // (of a CTA)
  static constexpr int NS = (BN / CTAS == 256) ? 4 : 6;               // stages
  static constexpr int SMEM = NS * STAGE_BYTES + 1024 /* alignment slack */ + 256 /* barriers */ + 8 * 2048 /* epilogue staging */ + BN * 16 /* column table */;
  static constexpr int TMEM_COLS = 2 * BN;                            // two accumulators
};

// The epilogue of 32 consecutive columns n .. n + nv - 1 of output row m (one thread).
// A&S 7.1.26 form of erf (absolute error below 2e-7, far inside the bf16 rounding of the correction it feeds)
__device__ __forceinline__ float gelu_quick(float z, int act) {
  if (act != TARDIS_ACT_GELU_ERF) return gelu_f32(z, act);
  const float x = fabsf(z) * 0.7071067811865476f;
  const float t = __fdividef(1.f, fmaf(0.3275911f, x, 1.f));
  float poly = fmaf(1.061405429f, t, -1.453152027f);
  poly = fmaf(poly, t, 1.421413741f);
  poly = fmaf(poly, t, -0.284496736f);
  poly = fmaf(poly, t, 0.254829592f);
  const float e = 1.f - poly * t * __expf(-x * x);          // erf(|z| / sqrt 2)
  return 0.5f * z * (1.f + copysignf(e, z));
}

// `stage`: 16 x 32 floats of shared memory of the calling warp (element [i][lane]); `tab`: the tile's column table (see
// fill_table), from column n on.
__device__ __forceinline__ void epilogue_chunk(const KParams& p, float (&v)[32], int m, int n, int nv, bool first_split, bool have_acc,
                                               float* stage, const float4* tab, int lane) {
  if (p.epilogue == GEMM_EPI_FLAGS) {
    // (the table holds lo - b1 and hi - b1: where the rounding of that difference could matter, |score - b1| and with it the
    // allowance is more than a hundred times as large, and the pair is re-evaluated)
    const float xn = p.rowscale[m];
    const uint32_t valid = nv == 32 ? 0xffffffffu : ((1u << nv) - 1u);
    uint32_t word = valid;                                   // a non-finite token: every neuron flagged
    if (xn <= 3.0e38f) {
      const float kx = p.keps * xn;
      uint32_t outside = 0u, open = 0u;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float4 t = tab[i];
        const float dl = v[i] - t.x, du = v[i] - t.y;
        outside |= (!(dl >= 0.f && du < 0.f) ? 1u : 0u) << i;
        open |= (fminf(fabsf(dl), fabsf(du)) <= fmaf(t.z, kx, 1e-30f) ? 1u : 0u) << i;
      }
      word = outside & valid;
      // (a token of zeros has no error, and its scores, the biases, may well lie on range ends)
      for (uint32_t w = xn > 0.f ? open & valid : 0u; w; w &= w - 1u) {      // rare
        const unsigned int slot = atomicAdd(&p.rcount[m], 1u);
        if (slot < (unsigned int)p.rcap) p.rlist[size_t(m) * p.rcap + slot] = uint32_t(n + __ffs(w) - 1);
      }
    }
    p.bitmap_out[size_t(m) * (p.N / 32) + (n >> 5)] = word;
    if (p.out_f32) {
      float* o = p.out_f32 + size_t(m) * p.ldo + n;
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < nv) o[i] = v[i] + tab[i].w;
    }
    return;
  }
  if (p.epilogue == GEMM_EPI_F32 && p.splits > 1) {
    float* o = p.out_f32 + size_t(m) * p.ldo + n;
    const bool with_bias = p.bias && first_split;
    if (have_acc || with_bias) {
      if (nv == 32 && (p.ldo & 3) == 0) {
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          float4 t = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
          if (with_bias) { t.x += p.bias[n + i]; t.y += p.bias[n + i + 1]; t.z += p.bias[n + i + 2]; t.w += p.bias[n + i + 3]; }
          asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(o + i), "f"(t.x), "f"(t.y), "f"(t.z), "f"(t.w) : "memory");
        }
      } else {
        for (int i = 0; i < nv; ++i) atomicAdd(o + i, v[i] + (with_bias ? p.bias[n + i] : 0.f));
      }
    }
  } else if (p.epilogue == GEMM_EPI_F32) {
    float* o = p.out_f32 + size_t(m) * p.ldo + n;
    if (nv == 32 && (p.ldo & 3) == 0) {
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        float4 t = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        if (p.bias) { t.x += p.bias[n + i]; t.y += p.bias[n + i + 1]; t.z += p.bias[n + i + 2]; t.w += p.bias[n + i + 3]; }
        *reinterpret_cast<float4*>(o + i) = t;
      }
    } else {
      for (int i = 0; i < nv; ++i) o[i] = v[i] + (p.bias ? p.bias[n + i] : 0.f);
    }
  } else {
    // bf16 outputs: this thread's 32 values become four 16-byte stores
    if (p.epilogue == GEMM_EPI_BF16) {
      const float* const bias = p.bias + n;
      if (nv == 32) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] += bias[i];
      } else {
        for (int i = 0; i < nv; ++i) v[i] += bias[i];
      }
    } else {   // GEMM_EPI_DELTA: one flag word covers this thread's 32 columns
      // Only the flagged tenth of the elements needs the activation, at different columns in every row.  The tanh form is evaluated for all of
      // them; for the others the accumulators go to shared memory, each thread walks the set bits of its own word, and the corrections
      // come back under the word's mask.
      uint32_t word = p.bitmap[size_t(m) * (p.N / 32) + (n >> 5)];
      if (nv < 32) word &= (1u << nv) - 1u;
      if (p.act == TARDIS_ACT_GELU_TANH) {
        // evaluated for every element, without branches: the walk over the set bits below waits for its row with the most of them, one
        // activation after the other (2048 x 16384 x 4096 with this epilogue 202 us, 210 with the walk, 173 with that of the flags)
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const float4 t = tab[i];
          const float z = v[i] + t.x, dl = gelu_tanh_f32(z) - t.y * z - t.z;
          v[i] = (word >> i) & 1u ? dl : 0.f;
        }
      } else
#pragma unroll
      for (int half = 0; half < 32; half += 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) stage[i * 32 + lane] = v[half + i];
        for (uint32_t w = (word >> half) & 0xffffu; w; w &= w - 1u) {
          const int i = __ffs(w) - 1;
          const float4 t = tab[half + i];
          const float z = stage[i * 32 + lane] + t.x;
          stage[i * 32 + lane] = gelu_quick(z, p.act) - t.y * z - t.z;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) v[half + i] = ((word >> (half + i)) & 1u) ? stage[i * 32 + lane] : 0.f;
      }
    }
    __nv_bfloat16* o = p.out_bf16 + size_t(m) * p.ldo + n;
    if (nv == 32 && (p.ldo & 7) == 0) {
#pragma unroll
      for (int i = 0; i < 32; i += 8) {
        __nv_bfloat162 h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(v[i + 2 * q], v[i + 2 * q + 1]);
        *reinterpret_cast<uint4*>(o + i) = *reinterpret_cast<const uint4*>(h);
      }
    } else {
      for (int i = 0; i < nv; ++i) o[i] = __float2bfloat16_rn(v[i]);
    }
  }
}

// What the epilogues look up per column, columns n0 .. n0 + count - 1 (one warp group of 128 threads): GEMM_EPI_FLAGS lo - bias,
// hi - bias, allowance per unit of |x|_1, bias; GEMM_EPI_DELTA bias, a, c.  (Looked up in global memory by every row of the tile,
// the scores of 2048 tokens on 4096 / 16384 took 427 us where the product alone takes 230.)
__device__ __forceinline__ void fill_table(const KParams& p, float4* tab, int n0, int count, int tid) {
  for (int c = tid; c < count; c += 128) {
    const int n = n0 + c;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n < p.N) {
      const float b = p.bias ? p.bias[n] : 0.f;
      if (p.epilogue == GEMM_EPI_DELTA) t = make_float4(b, p.a[n], p.c[n], 0.f);
      else {
        // a term of a score is at most max |code - zero-point| times the scale times |x|: 2 instead of 3 where the fold has found no 3
        const float most = p.second_used && p.bits == 2 && (p.second_used[n >> 7] & 2u) == 0u ? 2.f / 3.f : 1.f;
        t = make_float4(p.lo[n] - b, p.hi[n] - b, p.colscale[n] * most, b);
      }
    }
    tab[c] = t;
  }
}

// Persistent: CTA c works on tiles c, c + gridDim.x, ... of a banded raster.  Two accumulators in tensor memory:
// while the epilogue warps drain one, the MMA warp is already filling the other with the next tile.
//
// With CTAS = 2 two CTAs on neighbouring SMs share a tile of 256 x BN: each holds 128 rows of A and of the accumulator and half of the
// rows of B, and rank 0 issues the MMAs (M = 256) for both, so an operand row is written to and read from shared memory once
// per 256 rows of the other operand instead of once per 128 (a CTA of its own reads and writes 192 bytes of shared memory per clock at the
// MMAs' full rate, more than there are; 16384 prompt tokens of a 4096 / 16384 layer 7068 -> 6637 us, a calibration's product included
// 519 -> 497).  Rank 0's `full` barrier counts the bytes of both; a stage and an
// accumulator are handed back to both (multicast commit), and the accumulators of both have to be drained.
template <int BN, int CTAS>
__global__ void __launch_bounds__(NTHREADS, 1)
k_gemm(const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
       const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2, const KParams p) {
  using C = Cfg<BN, CTAS>;
  constexpr int TM = BM * CTAS, BROWS = BN / CTAS;      // rows of a tile; of B in this CTA
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::NS * C::STAGE_BYTES);
  uint64_t* empty = full + C::NS;
  uint64_t* accum_full = empty + C::NS;        // [2]
  uint64_t* accum_empty = accum_full + 2;      // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum_empty + 2);
  volatile uint32_t* failed = tmem_slot + 1;

  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp: uniform, and known to be)
  const int nm = (p.M + TM - 1) / TM, nn = (p.N + BN - 1) / BN;
  const int ntiles = nm * nn * p.splits;
  const int rank = CTAS == 2 ? int(cluster_rank()) : 0, first_tile = blockIdx.x / CTAS, step = gridDim.x / CTAS;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&accum_full[b], 1); mbar_init(&accum_empty[b], 8 * CTAS); }
    *failed = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA1) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB1) : "memory");
  }
  if (warp == 1) {                                     // the whole warp; a power of two >= 32 fp32 columns
    if (CTAS == 2) tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
    else tmem_alloc(tmem_slot, C::TMEM_COLS);
  }
  tc_fence_before();
  if (CTAS == 2) cluster_sync();                       // (the other CTA's barriers are reported to)
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // tile -> first row, first column, k-block range
  auto decode = [&](int tile, int& m0, int& n0, int& kb_lo, int& nkb, int& z) {
    z = tile / (nm * nn);
    const int rem = tile - z * (nm * nn);
    // raster: bands of `band` tiles along the dimension with fewer tiles, walked across the other dimension, so
    // that the CTAs running at the same time cover a compact block and share its operand tiles in L2
    const int F = p.fast_m ? nm : nn, S = p.fast_m ? nn : nm;
    const int bi = rem / (p.band * S), r2 = rem - bi * (p.band * S);
    const int w = min(p.band, F - bi * p.band);
    const int slow = r2 / w, fast = bi * p.band + (r2 - slow * w);
    const int mi = p.fast_m ? fast : slow, ni = p.fast_m ? slow : fast;
    m0 = mi * TM + rank * BM; n0 = ni * BN;
    int nkb_all = p.kb1;
    if (p.kb2 > 0) {
      bool used = p.second_used == nullptr;
      for (int r = n0; r < min(p.N, n0 + BN) && !used; r += 128) used = (__ldg(p.second_used + (r >> 7)) & 1u) != 0u;
      if (used) nkb_all += p.kb2;
    }
    const int per = (nkb_all + p.splits - 1) / p.splits;   // k blocks per split of the channel range
    kb_lo = z * per;
    nkb = max(0, min(nkb_all, kb_lo + per) - kb_lo);
  };

  int issued = 0;                                      // fills of a stage, by warp 0
  if (warp == 0) {
    // ---------------- TMA producer ----------------
    int s = 0, parity = 1;                             // stage and the phase of its `empty` barrier to wait for
    for (int tile = first_tile; tile < ntiles; tile += step) {
      int m0, n0, kb_lo, nkb, z;
      decode(tile, m0, n0, kb_lo, nkb, z);
      for (int kg = kb_lo; kg < kb_lo + nkb; ++kg) {   // k block in the whole channel range
        if (!mbar_wait_issue(&empty[s], parity, failed)) break;
        ++issued;
        const bool second = kg >= p.kb1;
        const int kx = (second ? kg - p.kb1 : kg) * BK;
        uint8_t* sa = smem + s * C::STAGE_BYTES;
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(&full[s], CTAS * C::STAGE_BYTES);
          if (CTAS == 2) {
            const uint32_t bar = in_rank_0(&full[s]);
            tma_load_2d_pair(sa, second ? &tmA2 : &tmA1, kx, m0, bar);
            tma_load_2d_pair(sa + BM * BK * 2, second ? &tmB2 : &tmB1, kx, n0 + rank * BROWS, bar);
          } else {
            tma_load_2d(sa, second ? &tmA2 : &tmA1, kx, m0, &full[s]);
            tma_load_2d(sa + BM * BK * 2, second ? &tmB2 : &tmB1, kx, n0, &full[s]);
          }
        }
        if (++s == C::NS) { s = 0; parity ^= 1; }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (of a pair: rank 0) ----------------
    constexpr uint32_t idesc = instr_desc_bf16(TM, BN);
    const uint64_t adesc = smem_desc_k_major_sw128(smem_u32(smem)), bdesc = smem_desc_k_major_sw128(smem_u32(smem) + BM * BK * 2);
    int s = 0, parity = 0;
    uint32_t use = 0;                                  // accumulator uses so far
    for (int tile = rank == 0 ? first_tile : ntiles; tile < ntiles; tile += step) {
      int m0, n0, kb_lo, nkb, z;
      decode(tile, m0, n0, kb_lo, nkb, z);
      if (nkb == 0) continue;                          // nothing to add: the epilogue takes zeros
      const uint32_t ab = use & 1u;
      // the epilogue warps have drained this accumulator's previous tile
      bool ok = mbar_wait_issue(&accum_empty[ab], ((use >> 1) & 1) ^ 1, failed);
      tc_fence_after();
      const uint32_t tacc = tmem_base + ab * BN;
      for (int kb = 0; kb < nkb; ++kb) {
        ok = mbar_wait_issue(&full[s], parity, failed);
        tc_fence_after();
        const uint64_t da = adesc + uint32_t(s * (C::STAGE_BYTES >> 4)), db = bdesc + uint32_t(s * (C::STAGE_BYTES >> 4));
        if (elect_one() && ok) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            if (CTAS == 2) umma_f16_pair(tacc, da + k * 2, db + k * 2, idesc, (kb | k) != 0 ? 1u : 0u);
            else umma_f16(tacc, da + k * 2, db + k * 2, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          if (CTAS == 2) umma_commit_pair(&empty[s]);  // frees the stage when these MMAs have read it
          else umma_commit(&empty[s]);
        }
        if (++s == C::NS) { s = 0; parity ^= 1; }
      }
      if (elect_one() && ok) {                         // accumulator complete
        if (CTAS == 2) umma_commit_pair(&accum_full[ab]);
        else umma_commit(&accum_full[ab]);
      }
      ++use;
    }
  } else {
    // ---------------- epilogue: a warp reads TMEM lanes 32 (warp % 4) .. + 31 and half of the columns ----------------
    const int q = warp & 3, half = (warp - 2) >> 2;
    uint8_t* const after = smem + C::NS * C::STAGE_BYTES + 256;
    float* const stage = reinterpret_cast<float*>(after) + (warp - 2) * 512;
    float4* const tab = reinterpret_cast<float4*>(after + 8 * 2048) + half * (BN / 2);
    const bool table = p.epilogue == GEMM_EPI_FLAGS || p.epilogue == GEMM_EPI_DELTA;
    uint32_t use = 0;
    bool ok = true;
    for (int tile = first_tile; tile < ntiles; tile += step) {
      int m0, n0, kb_lo, nkb, z;
      decode(tile, m0, n0, kb_lo, nkb, z);
      const int m = m0 + q * 32 + lane;
      const uint32_t ab = use & 1u;
      if (table) {                                         // (the warps of a half are a group of 128 threads)
        asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
        fill_table(p, tab, n0 + half * (BN / 2), BN / 2, (threadIdx.x - 64) & 127);
        asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
      }
      if (nkb > 0) {
        ok = ok && mbar_wait_warp(&accum_full[ab], (use >> 1) & 1);
        if (!ok) *failed = 1u;                               // (no way out here: the group meets at its barriers)
        tc_fence_after();
      }
      for (int ch = half * (BN / 64); ch < (half + 1) * (BN / 64); ++ch) {
        float v[32];
        if (nkb > 0) tmem_ld32(tmem_base + ab * BN + (uint32_t(q * 32) << 16) + uint32_t(ch * 32), v);
        else {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = 0.f;
        }
        const int n = n0 + ch * 32;
        const int nv = min(32, p.N - n);
        if (m < p.M && nv > 0) epilogue_chunk(p, v, m, n, nv, z == 0, nkb > 0, stage, tab + ch * 32 - half * (BN / 2), lane);   // (no early exit: tcgen05.ld needs the whole warp)
      }
      if (nkb > 0) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {                               // this warp's lanes of the accumulator may be overwritten
          if (CTAS == 2) mbar_arrive_cluster(in_rank_0(&accum_empty[ab]));
          else mbar_arrive(&accum_empty[ab]);
        }
        ++use;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *failed && p.error_word) atomicExch(p.error_word, 1ull);
  if (CTAS == 2) {
    // neither ends while the other may still report to it or its MMAs read it; copies of both report to rank 0
    if (threadIdx.x == 0 && rank == 1 && *failed) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_rank_0(const_cast<uint32_t*>(failed))), "r"(1u) : "memory");
    cluster_sync();
    if (rank == 0 && warp == 0 && *failed) land_copies<C::NS>(full, issued);
    if (warp == 1) tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
    cluster_sync();
  } else {
    if (warp == 0 && *failed) land_copies<C::NS>(full, issued);
    if (warp == 1) tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// ---- host side ------------------------------------------------------------------------------------------
template <int BN, int CTAS>
static tardis_status_t launch_bn(const GemmArgs& g, int dev, int sms, cudaStream_t s) {
  CUtensorMap a1, b1, a2, b2;
  if (!make_map(&a1, g.A1, g.M, g.K1, g.lda1, BM) || !make_map(&b1, g.B1, g.N, g.K1, g.ldb1, BN / CTAS)) return TARDIS_ERR_INVALID_ARG;
  a2 = a1; b2 = b1;
  if (g.K2 > 0 && (!make_map(&a2, g.A2, g.M, g.K2, g.lda2, BM) || !make_map(&b2, g.B2, g.N, g.K2, g.ldb2, BN / CTAS)))
    return TARDIS_ERR_INVALID_ARG;
  KParams p;
  p.M = g.M; p.N = g.N; p.kb1 = (g.K1 + BK - 1) / BK; p.kb2 = g.K2 > 0 ? (g.K2 + BK - 1) / BK : 0;
  p.second_used = g.second_used; p.epilogue = g.epilogue; p.ldo = g.ldo; p.act = g.act; p.splits = g.splits > 1 ? g.splits : 1;
  p.out_f32 = g.out_f32; p.out_bf16 = static_cast<__nv_bfloat16*>(g.out_bf16);
  p.bias = g.bias; p.a = g.a; p.c = g.c; p.bitmap = g.bitmap; p.error_word = g.error_word;
  p.lo = g.lo; p.hi = g.hi; p.colscale = g.colscale; p.rowscale = g.rowscale; p.keps = g.keps; p.bitmap_out = g.bitmap_out;
  p.rlist = g.rlist; p.rcount = g.rcount; p.rcap = g.rcap; p.bits = g.bits;
  static thread_local int room_on = -1;               // the device on which this thread last gave the kernel its shared memory
  if (dev != room_on) {
    TARDIS_CUDA_TRY(cudaFuncSetAttribute(k_gemm<BN, CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN, CTAS>::SMEM));
    room_on = dev;
  }
  const int nm = (g.M + BM * CTAS - 1) / (BM * CTAS), nn = (g.N + BN - 1) / BN;
  p.fast_m = nm <= nn ? 1 : 0;
  const int fcount = p.fast_m ? nm : nn;
  p.band = fcount <= 16 / (p.fast_m ? CTAS : 1) ? fcount : 12 / (p.fast_m ? CTAS : 1);
  const long tiles = long(nm) * nn * p.splits;
  const long at_once = sms / CTAS;                                    // one CTA per SM (shared memory), persistent
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(tiles < at_once ? tiles : at_once) * CTAS); cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = Cfg<BN, CTAS>::SMEM; cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CTAS; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = CTAS > 1 ? 1 : 0;
  TARDIS_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_gemm<BN, CTAS>, a1, b1, a2, b2, p));
  return TARDIS_OK;
}

}  // namespace gemm

tardis_status_t launch_gemm(const GemmArgs& g, cudaStream_t s) {
  using namespace gemm;
  if (g.M <= 0 || g.N <= 0 || g.K1 <= 0) return TARDIS_ERR_INVALID_ARG;
  if (!tensor_maps_available()) return TARDIS_ERR_UNSUPPORTED;
  auto bad = [](const void* p, int ld, int K) { return !p || (reinterpret_cast<uintptr_t>(p) & 15u) || (ld & 7) || (K & 7) || ld < K; };
  if (bad(g.A1, g.lda1, g.K1) || bad(g.B1, g.ldb1, g.K1)) return TARDIS_ERR_INVALID_ARG;
  if (g.K2 > 0 && (bad(g.A2, g.lda2, g.K2) || bad(g.B2, g.ldb2, g.K2))) return TARDIS_ERR_INVALID_ARG;
  if ((g.epilogue == GEMM_EPI_DELTA || g.epilogue == GEMM_EPI_FLAGS) && (g.N % 32)) return TARDIS_ERR_INVALID_ARG;
  if (g.epilogue == GEMM_EPI_FLAGS && !(g.bias && g.lo && g.hi && g.colscale && g.rowscale && g.bitmap_out && g.rlist && g.rcount))
    return TARDIS_ERR_INVALID_ARG;
  if (g.splits > 1 && g.epilogue != GEMM_EPI_F32) return TARDIS_ERR_INVALID_ARG;
  if (g.epilogue == GEMM_EPI_BF16 && !g.bias) return TARDIS_ERR_INVALID_ARG;
  // the epilogues store (or reduce) 16 bytes at a time
  auto misaligned = [](const void* p) { return p && (reinterpret_cast<uintptr_t>(p) & 15u); };
  if (misaligned(g.out_f32) || misaligned(g.out_bf16)) return TARDIS_ERR_INVALID_ARG;
  int dev = 0, sms = 0;
  TARDIS_CUDA_TRY(cudaGetDevice(&dev));
  TARDIS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // wide tiles when they still fill the machine (120 of 148 SMs), narrow ones for skinny problems
  const long splits = g.splits > 1 ? g.splits : 1, nm = (g.M + BM - 1) / BM, nn = (g.N + 255) / 256;
  if (nm * nn * splits * 100 < sms * 81) return launch_bn<128, 1>(g, dev, sms, s);
  // Pairs of CTAs unless the half tile that an odd number of row tiles leaves idle costs more, and for products of 2048 channels and more: a pair's
  // start, its two meetings and the accumulators' return to one of the two cost some 2 us and 1 us per wave.  us alone / in pairs, operands
  // from memory: 512 x 8192 (one wave) K = 1024 21.2 / 22.8, 2048 26.9 / 26.9, 4096 40.2 / 38.0; 512 x 16384 (two) 1024 32.3 / 33.0, 2048 46.2 / 42.5; 2048 x 16384
  // (seven) 512 93 / 103, 1024 100 / 105, 1536 118 / 119, 2048 152 / 138.  (With both operands in L2 and one wave the line lies at 6144: 2048 x 2048 x 4096 33.1 / 35.1,
  // 8192 59.7 / 56.6; weights that are read once per token or prompt come from memory.)
  const long waves = (nm * nn * splits + sms - 1) / sms, pair_waves = ((nm + 1) / 2 * nn * splits + sms / 2 - 1) / (sms / 2);
  const long blocks = (g.K1 + BK - 1) / BK + (g.K2 > 0 && !g.second_used ? (g.K2 + BK - 1) / BK : 0);
  const bool long_enough = blocks / splits >= 32;
  if (long_enough && pair_waves * 10 <= waves * 11) return launch_bn<256, 2>(g, dev, sms, s);
  return launch_bn<256, 1>(g, dev, sms, s);
}

}  // namespace tardis
