// The online path (Section 5.4) for fp32 layers: two launches, every product accumulated in fp64.
//
// Calls on such layers are small (256 / 1024 and 64 tokens: 50 MFLOP, 2.6 MB), so latency and launches are what counts; six
// launches of the generic kernels, the predictor among them with the tokens one after the other, took 284 us there.
//
//   k_f32_in: a CTA takes 32 neurons and 16 (or 8) tokens: predictor scores from the packed codes, flags, and the flagged pairs'
//     corrections, written to a dense [token][neuron] array (zero where not flagged).  Where its CTAs do not fill the SMs once, the exact
//     pre-activations of all pairs come out of the same walk over the channels: there is nothing to do but to wait, and the flagged
//     pairs alone, eight lanes a pair behind the flags, wait for another round of loads.  Where there are more, work counts (the fp64
//     unit, and from 1024 / 4096 on the bytes of W1): the flagged pairs alone, or a second walk in tiles where they are many.
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
struct State {
  float* delta; unsigned int* nfl;
  int clusters[2][MAX_SPLITS + 1];        // of k_f32_out with 8 and 16 tokens: clusters of so many CTAs that run at once
};

template <int TT, int PRODUCTS> struct Smem {
  union {
    // tokens of a pass and the next (padded: four channels x eight tokens in different banks); channel 16 w + 4 t + q in row 16 w + 4 q + t
    double xs[2][KC][TT + 4];
    double red[PRODUCTS][NWARP][TT][TM];  // the warps' sums
  };
};
template <int TT> struct OutSmem : Smem<TT, 1> {
  double total[TT][TM];                   // their sum
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
  template <int PRODUCTS> __device__ __forceinline__ void put(Smem<TT, PRODUCTS>& sm, int product, int warp, int g, int t) const {
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
template <int TT, int PRODUCTS> __device__ __forceinline__ double sum_of(const Smem<TT, PRODUCTS>& sm, int product, int t, int m) {
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
  template <int PRODUCTS> __device__ __forceinline__ void store(Smem<TT, PRODUCTS>& sm, int buffer) const {
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

// One walk over the channels for a CTA's neurons and tokens: the scores' products (SCORES), those of the exact pre-activations (EXACT),
// or both.  FIRST: x has not been waited for yet.  Ends with the last products read from shared memory still under way in other warps.
template <int BITS, int TT, bool SCORES, bool EXACT, bool FIRST, int PRODUCTS>
__device__ __forceinline__ void walk(const Params& p, Smem<TT, PRODUCTS>& sm, Acc<TT>& acc, Acc<TT>& accz) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * TM, t0 = blockIdx.y * TT, ng = p.d / p.G;
  Tokens<TT> x;
  // a thread expands four channels of four neurons (all of one group: groups are multiples of 16): s (q - zp), exact in fp64; and
  // takes the same of W1
  const int g = lane >> 2, t4 = lane & 3;
  uint32_t w[4];                                           // 4 BITS bits from `shift` on: the codes of channels 4 t4 ..
  const int half = min(12 * t4 / 16, 1);                   // 3-bit codes: the first of the two half-words that hold them
  const int shift = BITS == 2 ? 8 * t4 : (BITS == 3 ? 12 * t4 - 16 * half : (BITS == 4 ? 16 * (t4 & 1) : 0));
  float sc[4], zp[4];
  float4 w1[4];
  auto load_weights = [&](int k0) {
    const int kb = k0 + warp * 16, k = kb + t4 * 4;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const size_t j = j0 + 4 * g + m;
      if (SCORES) {
        sc[m] = zp[m] = 0.f;
        if (kb < p.d) {
          sc[m] = p.scale[j * ng + kb / p.G];
          zp[m] = float(p.zero[j * ng + kb / p.G]);
          const uint32_t* const row = p.codes + j * (size_t(p.d) * BITS / 32);
          if (BITS == 3) {                                 // (48 bits from a half-word on)
            const uint16_t* const at = reinterpret_cast<const uint16_t*>(row) + kb * 3 / 16 + half;
            w[m] = uint32_t(at[0]) | uint32_t(at[1]) << 16;
          } else {
            w[m] = row[kb * BITS / 32 + (BITS == 8 ? t4 : (BITS == 4 ? t4 >> 1 : 0))];
          }
        }
      }
      if (EXACT) w1[m] = k < p.d ? *reinterpret_cast<const float4*>(p.W1 + j * p.d + k) : make_float4(0.f, 0.f, 0.f, 0.f);   // (d: a multiple of 8)
    }
  };
  load_weights(0);
  if (FIRST) asm volatile("griddepcontrol.wait;" ::: "memory");   // (x may come from the launch before)
  x.load(p.x, p.d, p.n, t0, 0, p.d);
  int buffer = 0;
  for (int k0 = 0; k0 < p.d; k0 += KC, buffer ^= 1) {
    x.store(sm, buffer);
    double v[4][4], u[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (SCORES) {
        const double s = double(sc[m]), z = 4503599627370496.0 + double(zp[m]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {                      // channel 4 t4 + c
          const uint32_t q = (w[m] >> (shift + BITS * c)) & ((1u << BITS) - 1u);
          // (2^52 + q) - (2^52 + zp): the code as a double without a conversion
          v[c][m] = s * (__hiloint2double(0x43300000, int(q)) - z);
        }
      }
      if (EXACT) { u[0][m] = double(w1[m].x); u[1][m] = double(w1[m].y); u[2][m] = double(w1[m].z); u[3][m] = double(w1[m].w); }
    }
    __syncthreads();                                       // (a buffer is written again two passes on, behind this barrier)
    if (k0 + KC < p.d) { load_weights(k0 + KC); x.load(p.x, p.d, p.n, t0, k0 + KC, p.d); }
    if (SCORES) acc.multiply(v, &sm.xs[buffer][warp * 16], g, t4);
    if (EXACT) accz.multiply(u, &sm.xs[buffer][warp * 16], g, t4);
  }
}

// BOTH: scores and exact pre-activations in one walk; else the scores alone, and then, by the tile's number of flagged pairs, the
// flagged pairs one by one or a second walk.  A pair of its own takes four times the clocks of a pair of the second walk (two conversions
// per multiply-add and no reuse; 1024 / 4096 and 256 tokens: 6 us per hundredth of the pairs that is flagged, a second walk 146 us), so a
// quarter is where the second walk begins.  Registers: one CTA per SM is all there is for BOTH (1024 / 4096, 1 token 24.3 us with 174,
// 31.7 with the 128 of two); else two, as 80 hold back the loads (2048 / 8192, 1 token 60 us with 128, 77 with 80).
template <int BITS, int TT, bool BOTH>
__global__ void __launch_bounds__(NT, BOTH ? 1 : 2) k_f32_in(const Params p) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<TT, BOTH ? 2 : 1>& sm = *reinterpret_cast<Smem<TT, BOTH ? 2 : 1>*>(raw);
  __shared__ int pairs[BOTH ? 1 : TT * TM];
  __shared__ int npairs;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int j0 = blockIdx.x * TM, t0 = blockIdx.y * TT;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!BOTH && threadIdx.x == 0) npairs = 0;
  Acc<TT> acc = {}, accz = {};
  walk<BITS, TT, true, BOTH, true>(p, sm, acc, accz);
  __syncthreads();
  acc.put(sm, 0, warp, g, t4);
  if (BOTH) accz.put(sm, 1, warp, g, t4);
  __syncthreads();
  // scores -> flags -> corrections; lane = neuron, a warp takes tokens warp, warp + 8 (all at once: their fp64 chains overlap)
  const int j = j0 + lane;
  const double lo = double(p.lo[j]), hi = double(p.hi[j]), b1 = double(p.b1[j]), fa = double(p.a[j]), fc = double(p.c[j]);
  auto correction = [&](double z) { return float(gelu_f64(z, p.act) - fa * z - fc); };
  bool flag[TT / NWARP];
  float delta[TT / NWARP];
#pragma unroll
  for (int k = 0; k < TT / NWARP; ++k) {
    const int t = warp + k * NWARP;
    const double zhat = sum_of(sm, 0, t, lane) + b1;
    flag[k] = !(lo <= zhat && zhat < hi);
    if (BOTH) delta[k] = correction(sum_of(sm, 1, t, lane) + b1);
    if (p.dbg_scores && t0 + t < p.n) p.dbg_scores[size_t(t0 + t) * p.h + j] = zhat;
  }
#pragma unroll
  for (int k = 0; k < TT / NWARP; ++k) {
    const int t = t0 + warp + k * NWARP;
    if (t >= p.n) break;
    if (BOTH || !flag[k]) p.delta[size_t(t) * p.h + j] = BOTH && flag[k] ? delta[k] : 0.f;
    const uint32_t word = __ballot_sync(0xffffffffu, flag[k]);
    if (lane == 0 && word) atomicAdd(&p.nfl[t], (unsigned int)__popc(word));
    if (lane == 0 && p.dbg_bitmap) p.dbg_bitmap[size_t(t) * (p.h / 32) + blockIdx.x] = word;
    if (!BOTH) {
      int base = 0;
      if (lane == 0 && word) base = atomicAdd(&npairs, __popc(word));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (flag[k]) pairs[base + __popc(word & ((1u << lane) - 1u))] = (t - t0) * TM + lane;
    }
  }
  if constexpr (!BOTH) {
    __syncthreads();
    const int np = npairs;
    if (np > TT * TM / 4) {
      walk<BITS, TT, false, true, false>(p, sm, acc, accz);
      __syncthreads();
      accz.put(sm, 0, warp, g, t4);
      __syncthreads();
#pragma unroll
      for (int k = 0; k < TT / NWARP; ++k) {
        const int t = warp + k * NWARP;
        delta[k] = correction(sum_of(sm, 0, t, lane) + b1);
        if (t0 + t < p.n && flag[k]) p.delta[size_t(t0 + t) * p.h + j] = delta[k];
      }
      return;
    }
    // eight lanes a pair
    const int sub = lane & 7;
    for (int e0 = warp * 4; e0 < np; e0 += NWARP * 4) {
      const int e = e0 + (lane >> 3);
      const int pr = pairs[min(e, np - 1)], jj = j0 + (pr & (TM - 1)), t = t0 + pr / TM;
      const float* row = p.W1 + size_t(jj) * p.d;
      const float* xt = p.x + size_t(t) * p.d;
      double z0 = 0.0, z1 = 0.0, z2 = 0.0, z3 = 0.0;       // (four chains: the latency of one would be most of the time)
#pragma unroll 8
      for (int k = sub * 4; k < p.d; k += 32) {            // (d is a multiple of 8, rows are 16-byte aligned)
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
}

template <int TT>
__global__ void __launch_bounds__(NT) k_f32_out(const Params p) {
  extern __shared__ __align__(16) unsigned char raw[];
  OutSmem<TT>& sm = *reinterpret_cast<OutSmem<TT>*>(raw);
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
  for (int t = warp; t < TT; t += NWARP) sm.total[t][lane] = sum_of(sm, 0, t, lane);
  // the CTAs of the cluster share out the tile's outputs; each adds up the parts of its own, in order
  if (p.splits > 1) asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
  else __syncthreads();
  const int share = (TT * TM + p.splits - 1) / p.splits, end = min((z + 1) * share, TT * TM);
  for (int o = z * share + int(threadIdx.x); o < end; o += NT) {
    const int t = t0 + o / TM, i = i0 + o % TM;
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
template <int TT, bool BOTH> static Kernel in_kernel(int bits) {
  return bits == 2 ? k_f32_in<2, TT, BOTH> : (bits == 3 ? k_f32_in<3, TT, BOTH> : (bits == 4 ? k_f32_in<4, TT, BOTH> : k_f32_in<8, TT, BOTH>));
}

}  // namespace f32

using namespace f32;

namespace {
// a launch of k_f32_out in clusters of `size`, with one attribute at `attr`
cudaLaunchConfig_t out_config(dim3 grid, int size, cudaStream_t s, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(NT); cfg.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = 1; attr->val.clusterDim.y = 1; attr->val.clusterDim.z = unsigned(size);
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cfg;
}
// may start while the launch before it still runs
void overlapped(cudaLaunchAttribute* attr) {
  attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr->val.programmaticStreamSerializationAllowed = 1;
}
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
  auto room = [](Kernel k, size_t bytes) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)); };
  TARDIS_CUDA_TRY(room(in_kernel<16, true>(H->bits), sizeof(Smem<16, 2>)));
  TARDIS_CUDA_TRY(room(in_kernel<16, false>(H->bits), sizeof(Smem<16, 1>)));
  TARDIS_CUDA_TRY(room(k_f32_out<16>, sizeof(OutSmem<16>)));
  TARDIS_CUDA_TRY(room(in_kernel<8, true>(H->bits), sizeof(Smem<8, 2>)));
  TARDIS_CUDA_TRY(room(in_kernel<8, false>(H->bits), sizeof(Smem<8, 1>)));
  TARDIS_CUDA_TRY(room(k_f32_out<8>, sizeof(OutSmem<8>)));
  for (int size = 2; size <= MAX_SPLITS; ++size) {
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg = out_config(dim3(1, 1, size), size, nullptr, &attr);
    cfg.dynamicSmemBytes = sizeof(OutSmem<8>);
    TARDIS_CUDA_TRY(cudaOccupancyMaxActiveClusters(&S->clusters[0][size], k_f32_out<8>, &cfg));
    cfg.dynamicSmemBytes = sizeof(OutSmem<16>);
    TARDIS_CUDA_TRY(cudaOccupancyMaxActiveClusters(&S->clusters[1][size], k_f32_out<16>, &cfg));
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
  const int tiles = (p.n + TT - 1) / TT, in_ctas = p.h / TM * tiles;
  // us with both in one walk against scores first, there with a twentieth to a third of the pairs flagged: 256 / 1024, 64 tokens (128 CTAs) 18.5
  // against 19.7 .. 21.5; 512 / 2048, 16 tokens (64) 21.1, 25.2 .. 28.8; 768 / 3072, 24 tokens (192) 45.6, 36.9 .. 42.9; 1024 / 4096, 64
  // tokens (512) 119, 92 .. 104.
  const bool both = in_ctas <= H->num_sms;
  cudaLaunchAttribute attrs[2];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.h / TM, tiles); cfg.blockDim = dim3(NT); cfg.dynamicSmemBytes = both ? sizeof(Smem<TT, 2>) : sizeof(Smem<TT, 1>); cfg.stream = s;
  overlapped(&attrs[0]);
  cfg.attrs = attrs; cfg.numAttrs = 1;
  TARDIS_CUDA_TRY(cudaLaunchKernelEx(&cfg, both ? in_kernel<TT, true>(H->bits) : in_kernel<TT, false>(H->bits), p));
  cfg = out_config(dim3((p.d + TM - 1) / TM, tiles, p.splits), p.splits, s, &attrs[1]);
  cfg.dynamicSmemBytes = sizeof(OutSmem<TT>);
  cfg.attrs = attrs; cfg.numAttrs = p.splits > 1 ? 2 : 1;
  TARDIS_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_f32_out<TT>, p));
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
    // parts of the split product: as many as leave it one wave of clusters, at least one pass of KC channels each
    const int tt = p.n <= 8 ? 8 : 16, tiles = ((p.d + TM - 1) / TM) * ((p.n + tt - 1) / tt);
    const int passes = (p.d + KC - 1) / KC + (p.h + KC - 1) / KC;
    p.splits = 1;
    for (int size = 2; size <= MAX_SPLITS && size <= passes; ++size)
      if (tiles <= S->clusters[tt == 8 ? 0 : 1][size]) p.splits = size;
    const tardis_status_t st = tt == 8 ? launch_chunk<8>(H, p, s) : launch_chunk<16>(H, p, s);
    if (st != TARDIS_OK) return st;
    H->launches += 2;
  }
  return TARDIS_OK;
}

}  // namespace tardis
