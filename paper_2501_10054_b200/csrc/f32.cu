// The online path (Section 5.4) for fp32 layers: two launches, every product accumulated in fp64.
//
// Calls on such layers are small (256 / 1024 and 64 tokens: 50 MFLOP, 2.6 MB), so latency and launches are what counts; six
// launches of the generic kernels, the predictor among them with the tokens one after the other, took 284 us there.
//
//   k_f32_in: a CTA takes 32 neurons and 16 (or 4) tokens: predictor scores from the packed codes, flags, and for the flagged
//     pairs the exact pre-activation and its correction, written to a dense [token][neuron] array (zero where not flagged).
//   k_f32_out: y = b_f + [C ; W2^T]^T [x ; corrections], one product over d + h channels; its channel range is split over the
//     CTAs, partial sums go to places of their own, and the CTA that finishes a tile last adds them in order and writes y.
//
// Both products: a warp holds the 32 outputs x 16 tokens of the CTA (a thread 4 x 4) for every eighth channel of the range, so
// that four 128-bit reads of shared memory serve sixteen fp64 multiply-adds; the eight warps' sums meet in shared memory.
// Bound by the fp64 pipe beyond a few hundred tokens of the larger layers.
#include <string.h>

#include <algorithm>
#include <new>

#include "common.cuh"
#include "exact.cuh"

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
  double ws[KC][TM];                      // weights of a pass
  double xs[KC][TT + 2];                  // tokens of a pass (two values of padding: the stores of a half-warp spread over the banks)
  double red[NWARP][TT][TM];              // the warps' sums
};

template <int NTK> struct Acc { double v[4][NTK]; };

// one pass: every eighth channel (of nk) of the staged weights and tokens into the warp's 32 x 4 NTK outputs
template <int NTK> __device__ __forceinline__ void accumulate(Acc<NTK>& acc, const Smem<4 * NTK>& sm, int nk, int warp, int lane) {
  const int mo = (lane & 7) * 4, to = (lane >> 3) * NTK;
#pragma unroll 4
  for (int k = warp; k < nk; k += NWARP) {
    const double2 w0 = *reinterpret_cast<const double2*>(&sm.ws[k][mo]), w1 = *reinterpret_cast<const double2*>(&sm.ws[k][mo + 2]);
    const double w[4] = {w0.x, w0.y, w1.x, w1.y};
    double x[NTK];
    if (NTK == 4) {
      const double2 x0 = *reinterpret_cast<const double2*>(&sm.xs[k][to]), x1 = *reinterpret_cast<const double2*>(&sm.xs[k][to + 2]);
      x[0] = x0.x; x[1 % NTK] = x0.y; x[2 % NTK] = x1.x; x[3 % NTK] = x1.y;
    } else {
      x[0] = sm.xs[k][to];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int t = 0; t < NTK; ++t) acc.v[i][t] += w[i] * x[t];
  }
}

// the eight warps' sums -> red; afterwards sum_of gives an output's total (after a barrier)
template <int NTK> __device__ __forceinline__ void put(const Acc<NTK>& acc, Smem<4 * NTK>& sm, int warp, int lane) {
  const int mo = (lane & 7) * 4, to = (lane >> 3) * NTK;
#pragma unroll
  for (int t = 0; t < NTK; ++t)
#pragma unroll
    for (int i = 0; i < 4; i += 2) *reinterpret_cast<double2*>(&sm.red[warp][to + t][mo + i]) = make_double2(acc.v[i][t], acc.v[i + 1][t]);
}
template <int TT> __device__ __forceinline__ double sum_of(const Smem<TT>& sm, int t, int m) {
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) s += sm.red[w][t][m];
  return s;
}

// tokens t0 .. t0 + TT - 1 at channels k0 .. k0 + KC - 1 of a [n][ld] array (zero outside) -> xs
template <int TT> __device__ __forceinline__ void stage_tokens(Smem<TT>& sm, const float* __restrict__ src, size_t ld, int n, int t0, int k0, int kend) {
  for (int e = threadIdx.x; e < TT * KC; e += NT) {
    const int kk = e & (KC - 1), t = e / KC;
    sm.xs[kk][t] = (t0 + t < n && k0 + kk < kend) ? double(src[size_t(t0 + t) * ld + k0 + kk]) : 0.0;
  }
}

template <int BITS, int NTK>
__global__ void __launch_bounds__(NT) k_f32_in(const Params p) {
  constexpr int TT = 4 * NTK;
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT>& sm = *reinterpret_cast<Smem<TT>*>(raw);
  __shared__ int pairs[TT * TM];
  __shared__ int npairs;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * TM, t0 = blockIdx.y * TT, ng = p.d / p.G;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) npairs = 0;
  Acc<NTK> acc = {};
  bool waited = false;
  for (int k0 = 0; k0 < p.d; k0 += KC) {
    __syncthreads();
    {
      // a thread expands 16 channels (one group: groups are multiples of 16) of neuron `lane`: s (q - zp), exact in fp64
      const int j = j0 + lane, kb = k0 + warp * 16;
      if (kb < p.d) {
        const double s = double(p.scale[size_t(j) * ng + kb / p.G]), zp = 4503599627370496.0 + double(p.zero[size_t(j) * ng + kb / p.G]);
        const uint32_t* row = p.codes + size_t(j) * (size_t(p.d) * BITS / 32);
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (BITS != 3) {
#pragma unroll
          for (int q = 0; q < BITS / 2; ++q) w[q] = row[kb * BITS / 32 + q];
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const uint32_t q = BITS == 3 ? (kb + c < p.d ? stream_code(row, kb + c, 3) : 0u) : (w[c * BITS / 32] >> (c * BITS % 32)) & ((1u << BITS) - 1u);
          // (2^52 + q) - (2^52 + zp): the code as a double without a conversion
          const double v = __hiloint2double(0x43300000, int(q)) - zp;
          sm.ws[warp * 16 + c][lane] = kb + c < p.d ? s * v : 0.0;
        }
      } else {
#pragma unroll
        for (int c = 0; c < 16; ++c) sm.ws[warp * 16 + c][lane] = 0.0;
      }
    }
    if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }   // (x may come from the launch before)
    stage_tokens<TT>(sm, p.x, p.d, p.n, t0, k0, p.d);
    __syncthreads();
    accumulate<NTK>(acc, sm, min(KC, p.d - k0), warp, lane);
  }
  put<NTK>(acc, sm, warp, lane);
  __syncthreads();
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
    double z = 0.0;
#pragma unroll 4
    for (int k = sub * 4; k < p.d; k += 32) {              // (d is a multiple of 8, rows are 16-byte aligned)
      const float4 w = *reinterpret_cast<const float4*>(row + k), v = *reinterpret_cast<const float4*>(xt + k);
      z += double(w.x) * double(v.x);
      z += double(w.y) * double(v.y);
      z += double(w.z) * double(v.z);
      z += double(w.w) * double(v.w);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if (sub == 0 && e < np) {
      z += double(p.b1[jj]);
      p.delta[size_t(t) * p.h + jj] = float(gelu_f64(z, p.act) - double(p.a[jj]) * z - double(p.c[jj]));
    }
  }
}

template <int NTK>
__global__ void __launch_bounds__(NT) k_f32_out(const Params p) {
  constexpr int TT = 4 * NTK;
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT>& sm = *reinterpret_cast<Smem<TT>*>(raw);
  __shared__ bool last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = blockIdx.x * TM, t0 = blockIdx.y * TT, z = blockIdx.z;
  const int passes_d = (p.d + KC - 1) / KC, passes = passes_d + (p.h + KC - 1) / KC;   // C first, then W2^T
  const int from = int((long long)passes * z / p.splits), to = int((long long)passes * (z + 1) / p.splits);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  Acc<NTK> acc = {};
  bool waited = false;
  for (int ps = from; ps < to; ++ps) {
    const bool fold = ps < passes_d;
    const int k0 = (fold ? ps : ps - passes_d) * KC, kend = fold ? p.d : p.h;
    const float* m = fold ? p.C : p.W2T;                   // both [channel][output]
    __syncthreads();
    for (int e = threadIdx.x; e < KC * TM; e += NT) {
      const int i = e & (TM - 1), k = e / TM;
      sm.ws[k][i] = (k0 + k < kend && i0 + i < p.d) ? double(m[size_t(k0 + k) * p.d + i0 + i]) : 0.0;
    }
    if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }
    stage_tokens<TT>(sm, fold ? p.x : p.delta, fold ? p.d : p.h, p.n, t0, k0, kend);
    __syncthreads();
    accumulate<NTK>(acc, sm, min(KC, kend - k0), warp, lane);
  }
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
  put<NTK>(acc, sm, warp, lane);
  __syncthreads();
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

}  // namespace f32

using namespace f32;

tardis_status_t f32_prepare(Handle* H, cudaStream_t s) {
  H->f32 = nullptr;
  if (H->dtype != TARDIS_F32) return TARDIS_OK;
  State* S = new (std::nothrow) State();
  if (!S) return TARDIS_ERR_ALLOC;
  memset(S, 0, sizeof(*S));
  H->f32 = S;
  S->ndone = size_t((H->d + TM - 1) / TM) * (MAX_CHUNK / 4);
  const size_t bytes[3] = {size_t(MAX_CHUNK) * H->h * 4, size_t(MAX_PARTS) * H->d * 8, (S->ndone + MAX_CHUNK) * 4};
  void** ptrs[3] = {reinterpret_cast<void**>(&S->delta), reinterpret_cast<void**>(&S->part), reinterpret_cast<void**>(&S->words)};
  for (int i = 0; i < 3; ++i) {
    const cudaError_t e = dev_malloc(ptrs[i], bytes[i]);
    if (e != cudaSuccess) { set_last_error(e, "cudaMalloc"); cudaGetLastError(); f32_release(H); return TARDIS_ERR_ALLOC; }
    H->bytes_scratch += bytes[i];
  }
  TARDIS_CUDA_TRY(cudaMemsetAsync(S->words, 0, bytes[2], s));
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

template <int NTK> static tardis_status_t launch_chunk(const Handle* H, const Params& p, cudaStream_t s) {
  using Kernel = void (*)(Params);
  const Kernel in = H->bits == 2 ? k_f32_in<2, NTK> : (H->bits == 3 ? k_f32_in<3, NTK> : (H->bits == 4 ? k_f32_in<4, NTK> : k_f32_in<8, NTK>));
  const int tiles = (p.n + 4 * NTK - 1) / (4 * NTK);
  const dim3 grids[2] = {dim3(p.h / TM, tiles), dim3((p.d + TM - 1) / TM, tiles, p.splits)};
  const Kernel kernels[2] = {in, k_f32_out<NTK>};
  for (int i = 0; i < 2; ++i) {
    TARDIS_CUDA_TRY(cudaFuncSetAttribute(kernels[i], cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(Smem<4 * NTK>))));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grids[i]; cfg.blockDim = dim3(NT); cfg.dynamicSmemBytes = sizeof(Smem<4 * NTK>); cfg.stream = s;
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
    const int ntk = p.n <= 4 ? 1 : 4, tiles = ((p.d + TM - 1) / TM) * ((p.n + 4 * ntk - 1) / (4 * ntk));
    const int passes = (p.d + KC - 1) / KC + (p.h + KC - 1) / KC;
    p.splits = std::max(1, std::min({2 * H->num_sms / tiles, passes, MAX_PARTS / p.n, 64}));
    const tardis_status_t st = ntk == 1 ? launch_chunk<1>(H, p, s) : launch_chunk<4>(H, p, s);
    if (st != TARDIS_OK) return st;
    H->launches += 2;
  }
  return TARDIS_OK;
}

}  // namespace tardis
