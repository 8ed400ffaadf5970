// The online path (Section 5.4) for fp32 layers: two launches, every product accumulated in fp64.
//
// Calls on such layers are small (256 / 1024 and 64 tokens: 50 MFLOP, 2.6 MB), so latency and launches are what counts; six
// launches of the generic kernels, the predictor among them with the tokens one after the other, took 284 us there.
//
//   k_f32_in: a CTA takes 32 neurons and 16 (or 8) tokens: predictor scores from the packed codes and, in the same pass over the
//     channels, the exact pre-activations; flags, and the flagged pairs' corrections, written to a dense [token][neuron] array (zero
//     where not flagged).  (The pre-activations of the flagged pairs alone, eight lanes a pair behind the flags, wait for another round
//     of loads and for two conversions per multiply-add, which the tenth of the work does not make up for.)
//   k_f32_out: y = b_f + [C ; W2^T]^T [x ; corrections], one product over d + h channels; its channel range is split over the
//     CTAs of a cluster, which add their sums up through distributed shared memory, in order.  (Partial sums in global memory, a
//     counter and the CTA that finishes last: three dependent trips to L2.  With that and the pairs above 256 / 1024 took 21.8 us for
//     64 tokens, now 18.5.)
//
// The products run on the fp64 matrix instruction (m16n8k8: 5 multiply-adds per value read; one output and all tokens per
// thread, with the tokens broadcast from shared memory, is bound four times over by those reads).  A warp has 32 outputs and a
// slice of 16 of the 128 channels of a pass; weights go from global memory into registers, which are the A operand; the tokens,
// widened once, are read from shared memory as the B operand; the eight warps' sums meet in shared memory at the end.
#include <string.h>

#include <algorithm>
#include <new>

#include "common.cuh"
#include "ptx.cuh"

namespace tardis {
namespace f32 {

constexpr int NT = 256, NWARP = 8;
constexpr int KC = 128;                   // channels per pass through shared memory
constexpr int TM = 32;                    // outputs (neurons, columns) per CTA
constexpr int MAX_CHUNK = 256;            // tokens per pass of the two kernels
constexpr int MAX_SPLITS = 8;             // CTAs of a cluster (portable size)

struct Params {
  int n, d, h, G, act, splits;
  const uint32_t* codes; const float* scale; const uint8_t* zero;
  const float *lo, *hi, *a, *c, *b1, *bf, *W1, *W2T, *C;
  const float* x; float* y;
  float* delta;                           // [MAX_CHUNK][h]
  unsigned int* nfl;                      // flagged neurons per token
  unsigned long long* counters;
  uint32_t* dbg_bitmap; double* dbg_scores;
};
struct State { float* delta; unsigned int* nfl; };

template <int TT> struct Smem {
  union {
    // tokens of a pass and the next (padded: four channels x eight tokens in different banks); channel 16 w + 4 t + q in row 16 w + 4 q + t
    double xs[2][KC][TT + 4];
    double red[2][NWARP][TT][TM];         // the warps' sums of one or two products
  };
  double total[TT][TM];                   // their sum (k_f32_out)
};

// A warp's 32 outputs x TT tokens.  Output 4 g + m of the CTA's 32 is row g (m even) or g + 8 (m odd) of row tile m / 2.
template <int TT> struct Acc {
  double c[2][TT / 8][4];
  // channels of the slice: w[s][m] = weight of channel 4 t + s and output 4 g + m (x has the slice's channels in that order)
  __device__ __forceinline__ void multiply(const double (&w)[4][4], const double (*x)[TT + 4], int g, int t) {
#pragma unroll
    for (int k8 = 0; k8 < 2; ++k8)
#pragma unroll
      for (int nt = 0; nt < TT / 8; ++nt) {
        const double b0 = x[k8 * 8 + t][nt * 8 + g], b1 = x[k8 * 8 + t + 4][nt * 8 + g];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
          ptx::mma_f64(c[mt][nt], w[2 * k8][2 * mt], w[2 * k8][2 * mt + 1], w[2 * k8 + 1][2 * mt], w[2 * k8 + 1][2 * mt + 1], b0, b1);
      }
  }
  // the eight warps' sums of an output go where sum_of finds them (barriers before and after are the caller's)
  __device__ __forceinline__ void put(Smem<TT>& sm, int product, int warp, int g, int t) const {
#pragma unroll
    for (int nt = 0; nt < TT / 8; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        double* const at = &sm.red[product][warp][nt * 8 + 2 * t + e][4 * g];
        *reinterpret_cast<double2*>(at) = make_double2(c[0][nt][e], c[0][nt][2 + e]);
        *reinterpret_cast<double2*>(at + 2) = make_double2(c[1][nt][e], c[1][nt][2 + e]);
      }
  }
};
template <int TT> __device__ __forceinline__ double sum_of(const Smem<TT>& sm, int product, int t, int m) {
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) s += sm.red[product][w][t][m];
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
      const int e = q * NT + threadIdx.x, t = e % TT, k = e / TT, row = (k >> 2) * 16 + (k & 3);
      sm.xs[buffer][row][t] = double(v[q].x);
      sm.xs[buffer][row + 4][t] = double(v[q].y);
      sm.xs[buffer][row + 8][t] = double(v[q].z);
      sm.xs[buffer][row + 12][t] = double(v[q].w);
    }
  }
};

template <int BITS, int TT>
__global__ void __launch_bounds__(NT) k_f32_in(const Params p) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT>& sm = *reinterpret_cast<Smem<TT>*>(raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * TM, t0 = blockIdx.y * TT, ng = p.d / p.G;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  Acc<TT> acc = {}, accz = {};
  Tokens<TT> x;
  // a thread expands four channels of four neurons (all of one group: groups are multiples of 16): s (q - zp), exact in fp64; and
  // takes the same of W1
  const int g = lane >> 2, t4 = lane & 3;
  uint32_t w[4][BITS == 8 ? 4 : 2];
  float sc[4], zp[4];
  float4 w1[4];
  auto load_weights = [&](int k0) {
    const int kb = k0 + warp * 16, k = kb + t4 * 4;
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
      w1[m] = k < p.d ? *reinterpret_cast<const float4*>(p.W1 + j * p.d + k) : make_float4(0.f, 0.f, 0.f, 0.f);   // (d: a multiple of 8)
    }
  };
  load_weights(0);
  asm volatile("griddepcontrol.wait;" ::: "memory");       // (x may come from the launch before)
  x.load(p.x, p.d, p.n, t0, 0, p.d);
  int buffer = 0;
  for (int k0 = 0; k0 < p.d; k0 += KC, buffer ^= 1) {
    x.store(sm, buffer);
    double v[4][4], u[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const double s = double(sc[m]), z = 4503599627370496.0 + double(zp[m]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {                        // channel 4 t4 + c
        uint32_t q;
        if (BITS == 3) q = uint32_t((uint64_t(w[m][0]) | uint64_t(w[m][1]) << 32) >> (3 * (4 * t4 + c))) & 7u;
        else if (BITS == 2) q = (w[m][0] >> (8 * t4 + 2 * c)) & 3u;
        else if (BITS == 4) q = ((t4 & 2 ? w[m][1] : w[m][0]) >> (16 * (t4 & 1) + 4 * c)) & 15u;
        else q = ((t4 == 0 ? w[m][0] : (t4 == 1 ? w[m][1] : (t4 == 2 ? w[m][BITS == 8 ? 2 : 0] : w[m][BITS == 8 ? 3 : 0]))) >> (8 * c)) & 255u;
        // (2^52 + q) - (2^52 + zp): the code as a double without a conversion
        v[c][m] = s * (__hiloint2double(0x43300000, int(q)) - z);
      }
      u[0][m] = double(w1[m].x); u[1][m] = double(w1[m].y); u[2][m] = double(w1[m].z); u[3][m] = double(w1[m].w);
    }
    __syncthreads();                                       // (a buffer is written again two passes on, behind this barrier)
    if (k0 + KC < p.d) { load_weights(k0 + KC); x.load(p.x, p.d, p.n, t0, k0 + KC, p.d); }
    acc.multiply(v, &sm.xs[buffer][warp * 16], g, t4);
    accz.multiply(u, &sm.xs[buffer][warp * 16], g, t4);
  }
  __syncthreads();
  acc.put(sm, 0, warp, g, t4);
  accz.put(sm, 1, warp, g, t4);
  __syncthreads();
  // scores -> flags -> corrections; lane = neuron, a warp takes tokens warp, warp + 8 (all at once: their fp64 chains overlap)
  const int j = j0 + lane;
  const double lo = double(p.lo[j]), hi = double(p.hi[j]), b1 = double(p.b1[j]), fa = double(p.a[j]), fc = double(p.c[j]);
  bool flag[TT / NWARP];
  float delta[TT / NWARP];
#pragma unroll
  for (int k = 0; k < TT / NWARP; ++k) {
    const int t = warp + k * NWARP;
    const double zhat = sum_of<TT>(sm, 0, t, lane) + b1, z = sum_of<TT>(sm, 1, t, lane) + b1;
    flag[k] = !(lo <= zhat && zhat < hi);
    delta[k] = float(gelu_f64(z, p.act) - fa * z - fc);
    if (p.dbg_scores && t0 + t < p.n) p.dbg_scores[size_t(t0 + t) * p.h + j] = zhat;
  }
#pragma unroll
  for (int k = 0; k < TT / NWARP; ++k) {
    const int t = t0 + warp + k * NWARP;
    if (t >= p.n) break;
    p.delta[size_t(t) * p.h + j] = flag[k] ? delta[k] : 0.f;
    const uint32_t word = __ballot_sync(0xffffffffu, flag[k]);
    if (lane == 0 && word) atomicAdd(&p.nfl[t], (unsigned int)__popc(word));
    if (lane == 0 && p.dbg_bitmap) p.dbg_bitmap[size_t(t) * (p.h / 32) + blockIdx.x] = word;
  }
}

template <int TT>
__global__ void __launch_bounds__(NT) k_f32_out(const Params p) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT>& sm = *reinterpret_cast<Smem<TT>*>(raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = blockIdx.x * TM, t0 = blockIdx.y * TT, z = blockIdx.z;
  const int passes_d = (p.d + KC - 1) / KC, passes = passes_d + (p.h + KC - 1) / KC;   // C first, then W2^T
  const int from = int((long long)passes * z / p.splits), to = int((long long)passes * (z + 1) / p.splits);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  Acc<TT> acc = {};
  Tokens<TT> x;
  const int g = lane >> 2, t4 = lane & 3;
  float4 w[4];                                             // channels 16 warp + 4 t4 + s of outputs 4 g .. 4 g + 3
  auto load_weights = [&](int ps) {
    const bool fold = ps < passes_d;
    const int k0 = (fold ? ps : ps - passes_d) * KC, kend = fold ? p.d : p.h;
    const float* m = (fold ? p.C : p.W2T) + i0 + 4 * g;    // both [channel][output]; d is a multiple of 8
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + warp * 16 + 4 * t4 + q;
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
  __syncthreads();
  acc.put(sm, 0, warp, g, t4);
  __syncthreads();
#pragma unroll
  for (int t = warp; t < TT; t += NWARP) sm.total[t][lane] = sum_of<TT>(sm, 0, t, lane);
  // the CTAs of the cluster share out the tile's outputs; each adds up the parts of its own, in order
  if (p.splits > 1) asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
  else __syncthreads();
  const int share = TT * TM / p.splits;                    // (splits: a power of two)
  for (int e = int(threadIdx.x); e < share; e += NT) {
    const int o = z * share + e, t = t0 + o / TM, i = i0 + o % TM;
    const uint32_t at = uint32_t(__cvta_generic_to_shared(&sm.total[0][0] + o));
    double part[MAX_SPLITS];
#pragma unroll
    for (int q = 0; q < MAX_SPLITS; ++q)
      if (q < p.splits)
        asm volatile("{\n .reg .b32 a;\n mapa.shared::cluster.u32 a, %1, %2;\n ld.shared::cluster.f64 %0, [a];\n}" : "=d"(part[q]) : "r"(at), "r"(q) : "memory");
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < MAX_SPLITS; ++q)
      if (q < p.splits) s += part[q];
    if (t < p.n && i < p.d) p.y[size_t(t) * p.d + i] = float(s + double(p.bf[i]));
  }
  if (p.splits > 1) asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");   // (others may still read)
  if (blockIdx.x == 0 && z == 0 && threadIdx.x < TT && t0 + int(threadIdx.x) < p.n) {   // (once per token)
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
struct Sizes { size_t bytes[2]; };                         // delta, nfl
Sizes sizes(const Handle* H) { return {{size_t(MAX_CHUNK) * H->h * 4, MAX_CHUNK * 4}}; }
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
  const Sizes sz = sizes(H);
  const size_t (&bytes)[2] = sz.bytes;
  void** ptrs[2] = {reinterpret_cast<void**>(&S->delta), reinterpret_cast<void**>(&S->nfl)};
  for (int i = 0; i < 2; ++i) {
    const cudaError_t e = dev_malloc(ptrs[i], bytes[i]);
    if (e != cudaSuccess) { set_last_error(e, "cudaMalloc"); cudaGetLastError(); f32_release(H); return TARDIS_ERR_ALLOC; }
    H->bytes_scratch += bytes[i];
  }
  TARDIS_CUDA_TRY(cudaMemsetAsync(S->nfl, 0, bytes[1], s));
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
  void* ptrs[] = {S->delta, S->nfl};
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
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = unsigned(p.splits);
    cfg.attrs = attr; cfg.numAttrs = i == 1 && p.splits > 1 ? 2 : 1;
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
    p.delta = S->delta; p.nfl = S->nfl; p.counters = H->counters;
    p.dbg_bitmap = H->dbg_bitmap ? H->dbg_bitmap + size_t(t0) * (H->h / 32) : nullptr;
    p.dbg_scores = H->dbg_scores ? H->dbg_scores + size_t(t0) * H->h : nullptr;
    // parts of the split product: about two CTAs per SM, at least one pass of KC channels each, a power of two up to a cluster's CTAs
    const int tt = p.n <= 8 ? 8 : 16, tiles = ((p.d + TM - 1) / TM) * ((p.n + tt - 1) / tt);
    const int passes = (p.d + KC - 1) / KC + (p.h + KC - 1) / KC;
    p.splits = 1;
    while (p.splits < MAX_SPLITS && 2 * p.splits <= passes && 2 * p.splits * tiles <= 2 * H->num_sms) p.splits *= 2;
    const tardis_status_t st = tt == 8 ? launch_chunk<8>(H, p, s) : launch_chunk<16>(H, p, s);
    if (st != TARDIS_OK) return st;
    H->launches += 2;
  }
  return TARDIS_OK;
}

}  // namespace tardis
