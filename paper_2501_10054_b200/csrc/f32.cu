// The online path (Section 5.4) for fp32 layers: two launches, every product accumulated in fp64.
//
// Calls on such layers are small (256 / 1024 and 64 tokens: 50 MFLOP, 2.6 MB), so latency and launches are what counts; six
// launches of the generic kernels, the predictor among them with the tokens one after the other, took 284 us there.
//
//   k_f32_in: a CTA takes 32 neurons and 16 (or 8) tokens: predictor scores from the packed codes, flags, and for the flagged
//     pairs the exact pre-activation and its correction, written to a dense [token][neuron] array (zero where not flagged).
//   k_f32_out: y = b_f + [C ; W2^T]^T [x ; corrections], one product over d + h channels; its channel range is split over the
//     CTAs, partial sums go to places of their own, and the CTA that finishes a tile last adds them in order and writes y.
//
// Both products run on the fp64 matrix instruction (m16n8k8: 5 multiply-adds per value read; one output and all tokens per
// thread, with the tokens broadcast from shared memory, is bound four times over by those reads).  A warp has 32 outputs and a
// slice of 16 of the 128 channels of a pass; weights go from global memory into registers, which are the A operand; the tokens,
// widened once, are read from shared memory as the B operand; the eight warps' sums meet in shared memory at the end.
#include <string.h>

#include <algorithm>
#include <new>

#include "common.cuh"

namespace tardis {
namespace f32 {

constexpr int NT = 256, NWARP = 8;
constexpr int KC = 128;                   // channels per pass through shared memory
constexpr int TM = 32;                    // outputs (neurons, columns) per CTA
constexpr int MAX_CHUNK = 256;            // tokens per pass of the two kernels
constexpr int MAX_PARTS = 512;            // tokens times parts of the split product (the workspace is sized for this)

struct Params {
  int n, d, h, G, act, splits;
  const uint32_t* codes; const float* scale; const uint8_t* zero;
  const float *lo, *hi, *a, *c, *b1, *bf, *W1, *W2T, *C;
  const float* x; float* y;
  float* delta;                           // [MAX_CHUNK][h]
  double* part;                           // [splits][n][d]
  unsigned int *done, *nfl;               // finished parts per output tile; flagged neurons per token
  unsigned long long* counters;
  uint32_t* dbg_bitmap; double* dbg_scores;
};
struct State { float* delta; double* part; unsigned int* words; size_t ndone; };

template <int TT> struct Smem {
  union {
    double xs[2][KC][TT + 4];             // tokens of a pass and the next (padded: four channels x eight tokens in different banks)
    double red[NWARP][TT][TM];            // the warps' sums
  };
};

// D += A B, A 16 x 8 (rows: outputs), B 8 x 8 (columns: tokens).  With g = lane / 4, t = lane % 4: a0..a3 = A[g][t], A[g + 8][t],
// A[g][t + 4], A[g + 8][t + 4]; b0, b1 = B[t][g], B[t + 4][g]; c0..c3 = D[g][2t], D[g][2t + 1], D[g + 8][2t], D[g + 8][2t + 1].
__device__ __forceinline__ void mma_f64(double (&c)[4], double a0, double a1, double a2, double a3, double b0, double b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3]) : "d"(a0), "d"(a1), "d"(a2), "d"(a3), "d"(b0), "d"(b1));
}

// A warp's 32 outputs x TT tokens.  Output 4 g + m of the CTA's 32 is row g (m even) or g + 8 (m odd) of row tile m / 2.
template <int TT> struct Acc {
  double c[2][TT / 8][4];
  // channels of the slice: w[s][m] = weight of channel t + 4 s and output 4 g + m
  __device__ __forceinline__ void multiply(const double (&w)[4][4], const double (*x)[TT + 4], int g, int t) {
#pragma unroll
    for (int k8 = 0; k8 < 2; ++k8)
#pragma unroll
      for (int nt = 0; nt < TT / 8; ++nt) {
        const double b0 = x[k8 * 8 + t][nt * 8 + g], b1 = x[k8 * 8 + t + 4][nt * 8 + g];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
          mma_f64(c[mt][nt], w[2 * k8][2 * mt], w[2 * k8][2 * mt + 1], w[2 * k8 + 1][2 * mt], w[2 * k8 + 1][2 * mt + 1], b0, b1);
      }
  }
  // the eight warps' sums of an output meet (sum_of after this)
  __device__ __forceinline__ void put(Smem<TT>& sm, int warp, int g, int t) const {
    __syncthreads();
#pragma unroll
    for (int nt = 0; nt < TT / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        double* const at = &sm.red[warp][nt * 8 + 2 * t + e][4 * g];
        *reinterpret_cast<double2*>(at) = make_double2(c[0][nt][e], c[0][nt][2 + e]);
        *reinterpret_cast<double2*>(at + 2) = make_double2(c[1][nt][e], c[1][nt][2 + e]);
      }
    __syncthreads();
  }
};
template <int TT> __device__ __forceinline__ double sum_of(const Smem<TT>& sm, int t, int m) {
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) s += sm.red[w][t][m];
  return s;
}

// Tokens t0 .. t0 + TT - 1 at channels k0 .. k0 + KC - 1 of a [n][ld] array (zero outside): loaded into registers while the pass
// before is multiplied (a pass that waits for its own loads takes 3 us, mostly for them), then widened into xs.
template <int TT> struct Tokens {
  float4 v[TT * KC / 4 / NT];                              // token e % TT, channels 4 (e / TT) .. + 3
  __device__ __forceinline__ void load(const float* __restrict__ src, size_t ld, int n, int t0, int k0, int kend) {
#pragma unroll
    for (int q = 0; q < TT * KC / 4 / NT; ++q) {
      const int e = q * NT + threadIdx.x, t = e % TT, k = k0 + e / TT * 4;
      v[q] = (t0 + t < n && k < kend) ? *reinterpret_cast<const float4*>(src + size_t(t0 + t) * ld + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void store(Smem<TT>& sm, int buffer) const {
#pragma unroll
    for (int q = 0; q < TT * KC / 4 / NT; ++q) {
      const int e = q * NT + threadIdx.x, t = e % TT, k = e / TT * 4;
      sm.xs[buffer][k][t] = double(v[q].x);
      sm.xs[buffer][k + 1][t] = double(v[q].y);
      sm.xs[buffer][k + 2][t] = double(v[q].z);
      sm.xs[buffer][k + 3][t] = double(v[q].w);
    }
  }
};

template <int BITS, int TT>
__global__ void __launch_bounds__(NT) k_f32_in(const Params p) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT>& sm = *reinterpret_cast<Smem<TT>*>(raw);
  __shared__ int pairs[TT * TM];
  __shared__ int npairs;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * TM, t0 = blockIdx.y * TT, ng = p.d / p.G;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) npairs = 0;
  Acc<TT> acc = {};
  Tokens<TT> x;
  // a thread expands four channels of four neurons (all of one group: groups are multiples of 16): s (q - zp), exact in fp64
  const int g = lane >> 2, t4 = lane & 3;
  uint32_t w[4][BITS == 8 ? 4 : 2];
  float sc[4], zp[4];
  auto load_codes = [&](int k0) {
    const int kb = k0 + warp * 16;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const size_t j = j0 + 4 * g + m;
      sc[m] = zp[m] = 0.f;
      if (kb < p.d) {
        sc[m] = p.scale[j * ng + kb / p.G];
        zp[m] = float(p.zero[j * ng + kb / p.G]);
        const uint32_t* const row = p.codes + j * (size_t(p.d) * BITS / 32);
        if (BITS == 3) {                                   // 48 bits from a half-word on
          const uint16_t* at = reinterpret_cast<const uint16_t*>(row) + kb * 3 / 16;
          w[m][0] = uint32_t(at[0]) | uint32_t(at[1]) << 16;
          w[m][1] = at[2];
        } else {
#pragma unroll
          for (int q = 0; q < BITS / 2; ++q) w[m][q] = row[kb * BITS / 32 + q];
        }
      }
    }
  };
  load_codes(0);
  asm volatile("griddepcontrol.wait;" ::: "memory");       // (x may come from the launch before)
  x.load(p.x, p.d, p.n, t0, 0, p.d);
  int buffer = 0;
  for (int k0 = 0; k0 < p.d; k0 += KC, buffer ^= 1) {
    x.store(sm, buffer);
    double v[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const double s = double(sc[m]), z = 4503599627370496.0 + double(zp[m]);
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        const int c = q4 * 4;                              // channel c + t4
        uint32_t q;
        if (BITS == 3) q = uint32_t((uint64_t(w[m][0]) | uint64_t(w[m][1]) << 32) >> (3 * (c + t4))) & 7u;
        else q = (w[m][c * BITS / 32] >> ((c * BITS) % 32 + t4 * BITS)) & ((1u << BITS) - 1u);
        // (2^52 + q) - (2^52 + zp): the code as a double without a conversion
        v[q4][m] = s * (__hiloint2double(0x43300000, int(q)) - z);
      }
    }
    __syncthreads();                                       // (a buffer is written again two passes on, behind this barrier)
    if (k0 + KC < p.d) { load_codes(k0 + KC); x.load(p.x, p.d, p.n, t0, k0 + KC, p.d); }
    acc.multiply(v, &sm.xs[buffer][warp * 16], g, t4);
  }
  acc.put(sm, warp, g, t4);
  // scores -> flags; lane = neuron, a warp takes tokens warp, warp + 8, ...
  const int j = j0 + lane;
  const double lo = double(p.lo[j]), hi = double(p.hi[j]), b1 = double(p.b1[j]);
#pragma unroll
  for (int t = warp; t < TT; t += NWARP) {
    if (t0 + t >= p.n) break;
    const double zhat = sum_of<TT>(sm, t, lane) + b1;
    const bool flag = !(lo <= zhat && zhat < hi);
    const size_t at = size_t(t0 + t) * p.h + j;
    if (p.dbg_scores) p.dbg_scores[at] = zhat;
    if (!flag) p.delta[at] = 0.f;
    const uint32_t word = __ballot_sync(0xffffffffu, flag);
    int base = 0;
    if (lane == 0 && word) {
      base = atomicAdd(&npairs, __popc(word));
      atomicAdd(&p.nfl[t0 + t], (unsigned int)__popc(word));
    }
    if (lane == 0 && p.dbg_bitmap) p.dbg_bitmap[size_t(t0 + t) * (p.h / 32) + blockIdx.x] = word;
    base = __shfl_sync(0xffffffffu, base, 0);
    if (flag) pairs[base + __popc(word & ((1u << lane) - 1u))] = t * TM + lane;
  }
  __syncthreads();
  // exact pre-activations and corrections of the flagged pairs: eight lanes each
  const int np = npairs, sub = lane & 7;
  for (int e0 = warp * 4; e0 < np; e0 += NWARP * 4) {
    const int e = e0 + (lane >> 3);
    const int pr = pairs[min(e, np - 1)], jj = j0 + (pr & (TM - 1)), t = t0 + pr / TM;
    const float* row = p.W1 + size_t(jj) * p.d;
    const float* xt = p.x + size_t(t) * p.d;
    double z0 = 0.0, z1 = 0.0, z2 = 0.0, z3 = 0.0;         // (four chains: the latency of one would be most of the time)
#pragma unroll 8
    for (int k = sub * 4; k < p.d; k += 32) {              // (d is a multiple of 8, rows are 16-byte aligned)
      const float4 w = *reinterpret_cast<const float4*>(row + k), v = *reinterpret_cast<const float4*>(xt + k);
      z0 += double(w.x) * double(v.x);
      z1 += double(w.y) * double(v.y);
      z2 += double(w.z) * double(v.z);
      z3 += double(w.w) * double(v.w);
    }
    double z = (z0 + z1) + (z2 + z3);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if (sub == 0 && e < np) {
      z += double(p.b1[jj]);
      p.delta[size_t(t) * p.h + jj] = float(gelu_f64(z, p.act) - double(p.a[jj]) * z - double(p.c[jj]));
    }
  }
}

template <int TT>
__global__ void __launch_bounds__(NT) k_f32_out(const Params p) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT>& sm = *reinterpret_cast<Smem<TT>*>(raw);
  __shared__ bool last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = blockIdx.x * TM, t0 = blockIdx.y * TT, z = blockIdx.z;
  const int passes_d = (p.d + KC - 1) / KC, passes = passes_d + (p.h + KC - 1) / KC;   // C first, then W2^T
  const int from = int((long long)passes * z / p.splits), to = int((long long)passes * (z + 1) / p.splits);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  Acc<TT> acc = {};
  Tokens<TT> x;
  const int g = lane >> 2, t4 = lane & 3;
  float4 w[4];                                             // channels 16 warp + t4 + 4 s of outputs 4 g .. 4 g + 3
  auto load_weights = [&](int ps) {
    const bool fold = ps < passes_d;
    const int k0 = (fold ? ps : ps - passes_d) * KC, kend = fold ? p.d : p.h;
    const float* m = (fold ? p.C : p.W2T) + i0 + 4 * g;    // both [channel][output]; d is a multiple of 8
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + warp * 16 + t4 + 4 * q;
      w[q] = (k < kend && i0 + 4 * g < p.d) ? *reinterpret_cast<const float4*>(m + size_t(k) * p.d) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto load_tokens = [&](int ps) {
    const bool fold = ps < passes_d;
    x.load(fold ? p.x : p.delta, fold ? p.d : p.h, p.n, t0, (fold ? ps : ps - passes_d) * KC, fold ? p.d : p.h);
  };
  load_weights(from);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  load_tokens(from);
  int buffer = 0;
  for (int ps = from; ps < to; ++ps, buffer ^= 1) {
    x.store(sm, buffer);
    double v[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) { v[q][0] = double(w[q].x); v[q][1] = double(w[q].y); v[q][2] = double(w[q].z); v[q][3] = double(w[q].w); }
    __syncthreads();                                       // (a buffer is written again two passes on, behind this barrier)
    if (ps + 1 < to) { load_weights(ps + 1); load_tokens(ps + 1); }
    acc.multiply(v, &sm.xs[buffer][warp * 16], g, t4);
  }
  acc.put(sm, warp, g, t4);
  const int i = i0 + lane;
  if (p.splits > 1) {
#pragma unroll
    for (int t = warp; t < TT; t += NWARP)
      if (t0 + t < p.n && i < p.d) p.part[(size_t(z) * p.n + t0 + t) * p.d + i] = sum_of<TT>(sm, t, lane);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned int* const d = p.done + blockIdx.y * gridDim.x + blockIdx.x;
      last = atomicAdd(d, 1u) + 1u == (unsigned int)p.splits;
      if (last) *d = 0u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
  }
#pragma unroll
  for (int t = warp; t < TT; t += NWARP)
    if (t0 + t < p.n && i < p.d) {
      double s = 0.0;
      if (p.splits > 1) {
#pragma unroll 8
        for (int q = 0; q < p.splits; ++q) s += __ldcg(p.part + (size_t(q) * p.n + t0 + t) * p.d + i);
      } else {
        s = sum_of<TT>(sm, t, lane);
      }
      p.y[size_t(t0 + t) * p.d + i] = float(s + double(p.bf[i]));
    }
  if (blockIdx.x == 0 && threadIdx.x < TT && t0 + int(threadIdx.x) < p.n) {   // (once per token: the tile's last CTA)
    const unsigned int f = p.nfl[t0 + threadIdx.x];
    p.nfl[t0 + threadIdx.x] = 0u;
    if (f) {
      atomicAdd(&p.counters[CTR_FLAGGED_TOTAL], (unsigned long long)f);
      atomicMax(&p.counters[CTR_FLAGGED_MAX], (unsigned long long)f);
    }
  }
}

using Kernel = void (*)(Params);
template <int TT> static Kernel in_kernel(int bits) {
  return bits == 2 ? k_f32_in<2, TT> : (bits == 3 ? k_f32_in<3, TT> : (bits == 4 ? k_f32_in<4, TT> : k_f32_in<8, TT>));
}

}  // namespace f32

using namespace f32;

namespace {
// words per handle: finished parts per output tile, flagged neurons per token
size_t done_words(const Handle* H) { return size_t((H->d + TM - 1) / TM) * (MAX_CHUNK / 8); }
struct Sizes { size_t bytes[3]; };                         // delta, part, words
Sizes sizes(const Handle* H) { return {{size_t(MAX_CHUNK) * H->h * 4, size_t(MAX_PARTS) * H->d * 8, (done_words(H) + MAX_CHUNK) * 4}}; }
}  // namespace

size_t f32_room(const Handle* H) {
  size_t room = 0;
  for (size_t b : sizes(H).bytes) room += dev_room(b);
  return H->dtype == TARDIS_F32 ? room : 0;
}

tardis_status_t f32_prepare(Handle* H, cudaStream_t s) {
  H->f32 = nullptr;
  if (H->dtype != TARDIS_F32) return TARDIS_OK;
  State* S = new (std::nothrow) State();
  if (!S) return TARDIS_ERR_ALLOC;
  memset(S, 0, sizeof(*S));
  H->f32 = S;
  S->ndone = done_words(H);
  const Sizes sz = sizes(H);
  const size_t (&bytes)[3] = sz.bytes;
  void** ptrs[3] = {reinterpret_cast<void**>(&S->delta), reinterpret_cast<void**>(&S->part), reinterpret_cast<void**>(&S->words)};
  for (int i = 0; i < 3; ++i) {
    const cudaError_t e = dev_malloc(ptrs[i], bytes[i]);
    if (e != cudaSuccess) { set_last_error(e, "cudaMalloc"); cudaGetLastError(); f32_release(H); return TARDIS_ERR_ALLOC; }
    H->bytes_scratch += bytes[i];
  }
  TARDIS_CUDA_TRY(cudaMemsetAsync(S->words, 0, bytes[2], s));
  const Kernel wide[2] = {in_kernel<16>(H->bits), k_f32_out<16>}, narrow[2] = {in_kernel<8>(H->bits), k_f32_out<8>};
  for (int i = 0; i < 2; ++i) {
    TARDIS_CUDA_TRY(cudaFuncSetAttribute(wide[i], cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(Smem<16>))));
    TARDIS_CUDA_TRY(cudaFuncSetAttribute(narrow[i], cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(Smem<8>))));
  }
  return TARDIS_OK;
}

void f32_release(Handle* H) {
  State* S = static_cast<State*>(H->f32);
  if (!S) return;
  void* ptrs[] = {S->delta, S->part, S->words};
  for (void* q : ptrs)
    if (q) dev_free(q);
  delete S;
  H->f32 = nullptr;
}

template <int TT> static tardis_status_t launch_chunk(const Handle* H, const Params& p, cudaStream_t s) {
  const int tiles = (p.n + TT - 1) / TT;
  const dim3 grids[2] = {dim3(p.h / TM, tiles), dim3((p.d + TM - 1) / TM, tiles, p.splits)};
  const Kernel kernels[2] = {in_kernel<TT>(H->bits), k_f32_out<TT>};
  for (int i = 0; i < 2; ++i) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grids[i]; cfg.blockDim = dim3(NT); cfg.dynamicSmemBytes = sizeof(Smem<TT>); cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    TARDIS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernels[i], p));
  }
  return TARDIS_OK;
}

tardis_status_t launch_f32_forward(Handle* H, const void* xv, void* yv, int64_t n_total, cudaStream_t s) {
  State* S = static_cast<State*>(H->f32);
  for (int64_t t0 = 0; t0 < n_total; t0 += MAX_CHUNK) {
    Params p = {};
    p.n = int(std::min<int64_t>(n_total - t0, MAX_CHUNK)); p.d = H->d; p.h = H->h; p.G = H->G; p.act = H->act;
    p.codes = H->codes; p.scale = static_cast<const float*>(H->scale); p.zero = H->zero;
    p.lo = H->lo; p.hi = H->hi; p.a = H->a; p.c = H->c; p.b1 = H->b1; p.bf = H->bf;
    p.W1 = static_cast<const float*>(H->W1); p.W2T = static_cast<const float*>(H->W2T); p.C = static_cast<const float*>(H->C);
    p.x = static_cast<const float*>(xv) + size_t(t0) * H->d; p.y = static_cast<float*>(yv) + size_t(t0) * H->d;
    p.delta = S->delta; p.part = S->part; p.done = S->words; p.nfl = S->words + S->ndone; p.counters = H->counters;
    p.dbg_bitmap = H->dbg_bitmap ? H->dbg_bitmap + size_t(t0) * (H->h / 32) : nullptr;
    p.dbg_scores = H->dbg_scores ? H->dbg_scores + size_t(t0) * H->h : nullptr;
    // parts of the split product: about two CTAs per SM, at least one pass of KC channels each, what the workspace holds
    const int tt = p.n <= 8 ? 8 : 16, tiles = ((p.d + TM - 1) / TM) * ((p.n + tt - 1) / tt);
    const int passes = (p.d + KC - 1) / KC + (p.h + KC - 1) / KC;
    p.splits = std::max(1, std::min({2 * H->num_sms / tiles, passes, MAX_PARTS / p.n, 64}));
    const tardis_status_t st = tt == 8 ? launch_chunk<8>(H, p, s) : launch_chunk<16>(H, p, s);
    if (st != TARDIS_OK) return st;
    H->launches += 2;
  }
  return TARDIS_OK;
}

}  // namespace tardis
