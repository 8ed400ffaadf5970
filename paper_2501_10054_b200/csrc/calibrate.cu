// Offline statistics of a layer (Section 5.1, steps 2 and 3; the procedure is described with Insight 2 in Section 4.1): from the calibration pre-activations of every neuron,
// the range that holds the central portion of them (quantiles q_lo, q_hi) and the least-squares line
// y = a z + c of GELU over the samples inside that range.
//
// One CTA per neuron, the N samples in registers: the order statistics around the two quantiles are picked by a histogram, or,
// where that cannot tell them apart, by sorting (bitonic network over the next power of two, padded with +inf); the quantiles
// are interpolated in fp64 and rounded to fp32, and the regression sums run in fp64 in two passes (means, then centred
// second moments), GELU in fp64, once per sample.
#include <type_traits>

#include "common.cuh"

namespace tardis {
namespace cal {

constexpr int NT = 256;
constexpr int kMaxSamples = 8192;

// K sums over the CTA at once (one round of barriers); every thread gets them
template <int K> __device__ __forceinline__ void block_sums(double (&v)[K], double (&red)[K][NT / 32]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  __syncthreads();                                                        // red is free again
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[k][threadIdx.x >> 5] = v[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) t += red[k][w];
    v[k] = t;
  }
}

__device__ __forceinline__ double gelu_slope_f64(double z, int act) {
  if (act == TARDIS_ACT_RELU) return z > 0.0 ? 1.0 : 0.0;
  if (act == TARDIS_ACT_GELU_TANH) {
    const double k = 0.7978845608028654;
    const double u = k * (z + 0.044715 * z * z * z), t = tanh(u);
    return 0.5 * (1.0 + t) + 0.5 * z * (1.0 - t * t) * k * (1.0 + 3.0 * 0.044715 * z * z);
  }
  return 0.5 * (1.0 + erf(z * 0.7071067811865476)) + z * exp(-0.5 * z * z) * 0.3989422804014327;
}

// The activation by the formula that defines it, for decisions that rest on its exact values: where tanh is -1 (+1) to the last bit it
// is 0 (z), so that the errors of two ranges out there are both exactly 0 and the tie rule of the search applies.  (gelu_f64 keeps
// values of 1e-37 there: more exact, but another side then wins.)
__device__ __forceinline__ double activation_f64(double z, int act) {
  if (act != TARDIS_ACT_GELU_TANH) return gelu_f64(z, act);
  const double u = 0.7978845608028654 * (z + 0.044715 * z * z * z);
  return 0.5 * z * (1.0 + tanh(u));
}

// e^v as straight-line code, so that a thread's samples are evaluated side by side (exp branches, and its calls come one after the other):
// its Taylor series on |r| <= ln 2 / 2 (13 terms: 4e-18) times a power of two; v is taken into [-700, 700].
__device__ __forceinline__ double exp_straight(double v) {
  v = fmin(fmax(v, -700.0), 700.0);
  const double t = fma(v, 1.4426950408889634, 6755399441055744.0), k = t - 6755399441055744.0;   // the nearest whole number, in t's low bits
  const double r = fma(k, -2.3190468138462996e-17, fma(k, -0.6931471805599453, v));
  double p = 1.0 / 6227020800.0;                           // 1 / 13!
  p = fma(p, r, 1.0 / 479001600.0); p = fma(p, r, 1.0 / 39916800.0); p = fma(p, r, 1.0 / 3628800.0); p = fma(p, r, 1.0 / 362880.0);
  p = fma(p, r, 1.0 / 40320.0); p = fma(p, r, 1.0 / 5040.0); p = fma(p, r, 1.0 / 720.0); p = fma(p, r, 1.0 / 120.0);
  p = fma(p, r, 1.0 / 24.0); p = fma(p, r, 1.0 / 6.0); p = fma(p, r, 0.5); p = fma(p, r, 1.0); p = fma(p, r, 1.0);
  return __hiloint2double(__double2hiint(p) + (__double2loint(t) << 20), __double2loint(p));
}
// gelu_f64's tanh form likewise: z / (1 + e^-x), the reciprocal by two Newton steps from a float's; below x = -88 the result is 0, off by
// less than 1e-36.  (With exp and a division the activation took 7600 of a CTA's 23000 clocks in k_calibrate.)
__device__ __forceinline__ double gelu_tanh_f64(double z) {
  const double d = 1.0 + exp_straight(-1.5957691216057308 * (z + 0.044715 * z * z * z));
  float y0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(float(d)));
  double y = double(y0);
  y = fma(y, fma(-d, y, 1.0), y);
  y = fma(y, fma(-d, y, 1.0), y);
  return z * y;
}

// The n samples of neuron j plus its bias, NT E values over the CTA (+inf beyond n): thread t gets samples e NT + t.
template <int E> __device__ __forceinline__ void load_samples(float (&v)[E], const float* __restrict__ z, long long ldz,
                                                              const float* __restrict__ b1, int j, int n) {
  const float bias = b1 ? b1[j] : 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * NT + threadIdx.x;
    v[e] = i < n ? z[size_t(j) * ldz + i] + bias : __int_as_float(0x7f800000);
  }
}

// Ascending sort of the NT E values of the CTA; afterwards thread t holds positions t E .. t E + E - 1.  Bitonic network:
// strides below E stay inside a thread, strides below 32 E go by shuffle, and only the strides between warps (6 of the 66
// steps of 2048 values) pass through shared memory.  (All steps through shared memory: four times the time, bound by its
// bandwidth.)  sm: NT E floats.
__device__ __forceinline__ void order(float& x, float& y, bool up) {
  const float a = fminf(x, y), b = fmaxf(x, y);
  x = up ? a : b;
  y = up ? b : a;
}
template <int E> __device__ __forceinline__ void sort_samples(float (&v)[E], float* sm) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int k = 2; k <= E; k <<= 1)
#pragma unroll
    for (int s = k >> 1; s > 0; s >>= 1)
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (!(e & s)) order(v[e], v[e | s], ((tid * E + e) & k) == 0);
  for (int k = 2; k <= NT; k <<= 1) {                  // runs of k E values
    const bool up = (tid & k) == 0;
    int m = k >> 1;
    for (; m >= 32; m >>= 1) {
      const bool keep_min = ((tid & m) == 0) == up;
#pragma unroll
      for (int e = 0; e < E; ++e) sm[e * NT + tid] = v[e];
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float o = sm[e * NT + (tid ^ m)];
        v[e] = keep_min ? fminf(v[e], o) : fmaxf(v[e], o);
      }
      __syncthreads();
    }
    for (; m >= 1; m >>= 1) {
      const bool keep_min = ((tid & m) == 0) == up;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float o = __shfl_xor_sync(0xffffffffu, v[e], m);
        v[e] = keep_min ? fminf(v[e], o) : fmaxf(v[e], o);
      }
    }
#pragma unroll
    for (int s = E >> 1; s > 0; s >>= 1)
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (!(e & s)) order(v[e], v[e | s], up);
  }
}

// Least squares of the activation over the samples with l <= z < u (fp64, two passes: means, then centred second
// moments); thread 0 writes the line of neuron j; fewer than two samples in range: the tangent at the midpoint.
// gs: activation values of the thread's samples where they are in range.
template <int E> __device__ __forceinline__ void fit_and_store(const float (&v)[E], const double (&gs)[E], float lo_f, float hi_f, int act, int j,
                                                               float* __restrict__ lo, float* __restrict__ hi, float* __restrict__ a, float* __restrict__ c) {
  __shared__ double red3[3][NT / 32];
  __shared__ double red2[2][NT / 32];
  const double l = double(lo_f), u = double(hi_f);
  double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double x = double(v[e]);
    if (x >= l && x < u) { s[0] += 1.0; s[1] += x; s[2] += gs[e]; }
  }
  block_sums<3>(s, red3);
  const double cnt = s[0], safe = cnt > 0.0 ? cnt : 1.0;
  const double mz = s[1] / safe, ms = s[2] / safe;
  double m[2] = {0.0, 0.0};
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double x = double(v[e]);
    if (x >= l && x < u) { const double dz = x - mz; m[0] += dz * dz; m[1] += dz * (gs[e] - ms); }
  }
  block_sums<2>(m, red2);
  const double var = m[0] / safe, cov = m[1] / safe;
  if (threadIdx.x == 0) {
    double aj, cj;
    if (cnt >= 2.0 && var > 1e-30) { aj = cov / var; cj = ms - aj * mz; }
    else {                                             // too few samples in range: tangent at the midpoint
      const double mid = 0.5 * (l + u);
      aj = gelu_slope_f64(mid, act);
      cj = gelu_f64(mid, act) - aj * mid;
    }
    lo[j] = lo_f; hi[j] = hi_f; a[j] = float(aj); c[j] = float(cj);
  }
}

// The order statistics at four ranks (0 <= rank[q] < n) of the CTA's samples, without sorting them: a histogram over 1024 equal
// steps of their span tells which step holds a rank, and the few samples of that step are ranked among themselves.  (The step of a
// sample is a monotone function of its value, so the outcome is exact.)  False, the same for all threads, when a step holds too
// many (samples far out stretch the span) or the span is not finite: then the caller sorts.
constexpr int kSteps = 1024, kPick = 64;
template <int E> __device__ __forceinline__ bool pick_ranks(const float (&v)[E], int n, const int (&rank)[4], float (&stat)[4]) {
  __shared__ int hist[kSteps];
  __shared__ float picked[4][kPick];
  __shared__ int npicked[4], bin_at[4], before[4];
  __shared__ float lo_hi[2][NT / 32];
  __shared__ float result[4];
  __shared__ int wsum[NT / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float mn = __int_as_float(0x7f800000), mx = -mn;
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (e * NT + tid < n) { mn = fminf(mn, v[e]); mx = fmaxf(mx, v[e]); }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o)); mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o)); }
  if (lane == 0) { lo_hi[0][warp] = mn; lo_hi[1][warp] = mx; }
  for (int i = tid; i < kSteps; i += NT) hist[i] = 0;
  if (tid < 4) npicked[tid] = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) { mn = fminf(mn, lo_hi[0][w]); mx = fmaxf(mx, lo_hi[1][w]); }
  const float span = mx - mn, inv = float(kSteps) / span;
  if (!(span > 1e-30f && span < 1e30f)) return false;      // (all samples equal, too)
  int bin[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    bin[e] = e * NT + tid < n ? min(int((v[e] - mn) * inv), kSteps - 1) : -1;
    if (bin[e] >= 0) atomicAdd(&hist[bin[e]], 1);
  }
  __syncthreads();
  // a thread has kSteps / NT steps: running sums over the CTA
  constexpr int PER = kSteps / NT;
  int own[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) { own[i] = hist[tid * PER + i]; sum += own[i]; }
  int scan = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, scan, o); if (lane >= o) scan += t; }
  if (lane == 31) wsum[warp] = scan;
  __syncthreads();
  int from = scan - sum;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) if (w < warp) from += wsum[w];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (rank[q] >= from && rank[q] < from + own[i]) { bin_at[q] = tid * PER + i; before[q] = from; }
    from += own[i];
  }
  __syncthreads();
  const int want[4] = {bin_at[0], bin_at[1], bin_at[2], bin_at[3]};
#pragma unroll
  for (int e = 0; e < E; ++e)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (bin[e] == want[q]) {
        const int at = atomicAdd(&npicked[q], 1);
        if (at < kPick) picked[q][at] = v[e];
      }
  __syncthreads();
  if (max(max(npicked[0], npicked[1]), max(npicked[2], npicked[3])) > kPick) return false;
  if (warp < 4) {
    const int m = npicked[warp], r = rank[warp] - before[warp];
    for (int i = lane; i < m; i += 32) {
      const float x = picked[warp][i];
      int below = 0;
      for (int k = 0; k < m; ++k) { const float y = picked[warp][k]; below += (y < x || (y == x && k < i)) ? 1 : 0; }
      if (below == r) result[warp] = x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) stat[q] = result[q];
  return true;
}

// Bound by the latency of its barriers and by the fp64 activation.  16384 neurons x 2048 samples: 0.24 ms (0.28 with five CTAs per SM, two passes
// and an activation that branches, 0.46 ms with the
// samples sorted in registers, 0.91 ms with every step of the sort in shared memory and the activation as a fp64 tanh, evaluated twice).
// ERF: the erf form, which branches and is left out where nothing is inside, as beyond n (8192 x 1500: 152 us evaluated everywhere, 130); the
// others are straight on for every sample.
template <int E, bool ERF> __global__ void __launch_bounds__(NT, E <= 8 ? 6 : 1)   // (CTAs per SM: their barriers and chains overlap; one pass and no stored activations leave the registers for six)
k_calibrate(const float* __restrict__ z, long long ldz, const float* __restrict__ b1, int n, double q_lo, double q_hi,
            int act, float* __restrict__ lo, float* __restrict__ hi, float* __restrict__ a, float* __restrict__ c) {
  extern __shared__ float keys[];                      // [NT E]
  __shared__ float found[4];                           // the order statistics around the two quantiles
  __shared__ double red5[5][NT / 32];
  const int j = blockIdx.x, tid = threadIdx.x;
  float v[E];
  load_samples<E>(v, z, ldz, b1, j, n);
  // quantile at level q: between the order statistics around position q (n - 1)
  int rank[4];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    rank[2 * r] = int(floor((r == 0 ? q_lo : q_hi) * double(n - 1)));
    rank[2 * r + 1] = min(rank[2 * r] + 1, n - 1);
  }
  float stat[4];
  if (!pick_ranks<E>(v, n, rank, stat)) {
    sort_samples<E>(v, keys);
#pragma unroll
    for (int e = 0; e < E; ++e)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (tid * E + e == rank[q]) found[q] = v[e];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) stat[q] = found[q];
  }
  float range[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const double pos = (r == 0 ? q_lo : q_hi) * double(n - 1);
    const double w = pos - floor(pos);
    range[r] = float(__dadd_rn(__dmul_rn(double(stat[2 * r]), 1.0 - w), __dmul_rn(double(stat[2 * r + 1]), w)));
  }
  // Least squares of the activation over the samples inside, in one pass: moments about one of those samples, so that samples that are
  // all equal give a variance of exactly zero (the offset of the mean costs at most log10(n) digits of 16, with one sample far below all others).  Two passes (means first) need a
  // second round of barriers, and the activations kept in registers, which are then too many for a sixth CTA per SM.
  const float l = range[0], u = range[1];
  const double c0 = double(stat[1] >= l && stat[1] < u ? stat[1] : l);
  const double g0 = double(gelu_f32(float(c0), act));      // (near the activation there, for the same reason)
  double m[5] = {0.0, 0.0, 0.0, 0.0, 0.0};                 // count, y, g, y y, y g; y = z - c0, g = activation - g0
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool inside = v[e] >= l && v[e] < u;
    const double x = double(inside ? v[e] : float(c0));
    const double g = (ERF ? (inside ? gelu_f64(x, TARDIS_ACT_GELU_ERF) : g0) : (act == TARDIS_ACT_GELU_TANH ? gelu_tanh_f64(x) : gelu_f64(x, act))) - g0, y = x - c0;
    if (inside) { m[0] += 1.0; m[1] += y; m[2] += g; m[3] = fma(y, y, m[3]); m[4] = fma(y, g, m[4]); }
  }
  block_sums(m, red5);
  if (tid == 0) {
    const double cnt = m[0], safe = cnt > 0.0 ? cnt : 1.0, my = m[1] / safe, mg = m[2] / safe;
    const double var = m[3] / safe - my * my, cov = m[4] / safe - my * mg;
    double aj, cj;
    if (cnt >= 2.0 && var > 1e-30) { aj = cov / var; cj = (g0 + mg) - aj * (c0 + my); }
    else {                                                 // too few samples in range: tangent at the midpoint
      const double mid = 0.5 * (double(l) + double(u));
      aj = gelu_slope_f64(mid, act);
      cj = gelu_f64(mid, act) - aj * mid;
    }
    lo[j] = l; hi[j] = u; a[j] = float(aj); c[j] = float(cj);
  }
}

// ---- the greedy range search of Algorithm 1 (Section 5.1.1, "Range Searching") --------------------------------------
// One CTA per neuron.  (1) Sort the samples.  (2) Centroid: the sample with the highest Gaussian kernel density estimate
// (width 1.06 std N^-1/5, density evaluated at the samples, fp64).  (3) The greedy loop: range = centroid - k_l step ..
// centroid + k_r step, grown by one step on the side whose candidate range has the smaller error (right on ties; a side that
// has passed the outermost sample is not grown) until the share of samples inside reaches the neuron's threshold.  The error
// of a candidate is the mean squared residual of the least-squares line over the samples inside.  (4) The line over the
// final range, as in k_calibrate.
//
// Neither the densities nor the errors are needed as numbers, only which one is the largest / smaller, so both are screened
// by cheap values with a bound on what these can be off by, and evaluated as defined only where the bound leaves it open:
//   * density: the samples fall into bins of a quarter of the kernel width (only those that hold any are kept: some 130 of 260
//     possible ones); from the moments of the bins around it, each bin gets the Taylor polynomial of the density about its
//     centre (Hermite polynomials, order 4 on both sides), which gives all samples' densities to 1e-5 N.  Only the samples within
//     that of the best (some 30 of 2048) are looked at more closely: where they lie within a quarter of the kernel width, as they do
//     around a single mode, one pass over the samples in fp64 gives the density's expansion about their middle and with it all their
//     densities to 1e-12 N; else sums of exponentials in fp32 leave a handful.  What is left (almost always one) is evaluated in fp64.
//     All N^2 exponentials in fp64 took 95 % of the time at first, the fp32 sums and the fp64 ones after them a quarter.
//   * candidate errors: from moments of the samples that the steps on either side add (fp64, made for all steps at once and summed
//     up by scans).  The threads hold the errors of all ranges that the next 21 steps can lead to and decide for each what would be done
//     from it, so that the chain of dependent fp64 instructions is paid once per 21 steps and the walk itself is a look per step (by
//     one warp, six steps ahead and with the decisions made along the way, it was 40 % of the search).  Two errors closer than the
//     rounding bound of the moments (or moments that cancel) are evaluated by the definition; exact zeros of piecewise-linear activations, on
//     which the tie rule depends, thus stay exact.
// 16384 neurons x 2048 samples: 1.5 ms (2.5 before the expansion about the candidates' middle, the bins' sums without atomics and the
// walk of all threads; 133 ms with every density and error evaluated as defined).
constexpr int kMaxSearchSamples = 2048;
constexpr int kMaxSteps = 128;           // steps on one side whose moments are made at once, a thread per step and side
constexpr int kSeries = 10;              // terms of the density about the middle of the candidates
constexpr int kAhead = 21;               // steps that the CTA looks ahead: 253 ranges, one per thread
// Bins: samples within 5 standard deviations fill at most 10 / (0.25 * 1.06 N^-0.2) = 174 of them at N = 2048 (fewer below), and at
// most N / 25 samples lie beyond.
constexpr int kMaxBins = 272;

__device__ __forceinline__ float ex2f(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct Bins {
  float centre[kMaxBins];                // from the smallest sample on
  float m[5][kMaxBins];                  // sum of offset^n / n! of the bin's samples, offsets from the centre in kernel widths
  float l[5][kMaxBins];                  // Taylor coefficients of the density about the centre
  int start[kMaxBins + 1];               // position of the bin's first sample
};
struct Ahead {                           // of the ranges that the next steps can lead to
  double err[NT];
  float off[NT];
  uint16_t next[NT];                     // number of the range that follows, what is done (two bits), steps from the first one
};
struct Steps {
  double m[2][5][kMaxSteps + 1];         // [side][moment][k]: what the first k steps add
  int end[2][kMaxSteps + 1];             // position of the range's end after k steps
};

// Position of the highest density among the sorted samples (the smallest position among equals); the whole CTA, every thread gets
// it.  v: the thread's samples (positions tid E ...), keys: all of them; bw: kernel width (> 0); list: room for n positions.
template <int E> __device__ __forceinline__ int densest_sample(const float (&v)[E], const float* keys, int n, double bw, Bins& bins, int* list) {
  __shared__ float wmax[NT / 32];
  __shared__ int wcnt[NT / 32];
  __shared__ double bestv[NT / 32];
  __shared__ int besti[NT / 32];
  __shared__ int count;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float zmin = keys[0], zmax = keys[n - 1], inv = float(1.0 / bw), width = float(0.25 * bw);
  bool screen = bw > 1e-30 && bw < 1e30 && double(zmax) - double(zmin) < 1e30;
  // bins: a sample opens one where its predecessor is in another
  auto bin_of = [&](float z) { return floorf((z - zmin) * (4.f * inv)); };
  int first[E], nopen = 0;               // ordinal of the bin within the thread's samples
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = tid * E + e;
    if (i < n && (i == 0 || bin_of(v[e]) != bin_of(e ? v[e > 0 ? e - 1 : 0] : keys[i - 1]))) ++nopen;
    first[e] = nopen;
  }
  int scan = nopen;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, scan, o); if (lane >= o) scan += t; }
  if (lane == 31) wcnt[warp] = scan;
  if (tid == 0) count = 0;
  __syncthreads();
  int before = scan - nopen, nbins = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) { if (w < warp) before += wcnt[w]; nbins += wcnt[w]; }
  screen = screen && nbins <= kMaxBins;
  if (screen) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = tid * E + e, b = before + first[e] - 1;
      if (i < n && first[e] != (e ? first[e > 0 ? e - 1 : 0] : 0)) {
        // (distances from the smallest sample, which are exact or rounded to 2^-24 of themselves: a centre in the samples' own
        // coordinates would be off by an ulp of them, a fifth of the kernel width where the samples lie 4 ulps apart)
        bins.start[b] = i;
        bins.centre[b] = (bin_of(v[e]) + 0.5f) * width;
      }
    }
    if (tid == 0) bins.start[nbins] = n;
    __syncthreads();
    // moments: a pair of lanes adds up a bin's samples (runs of a thread's own samples added to the bins atomically: 10000 clocks)
    for (int b0 = 0; b0 < nbins; b0 += NT / 2) {
      const int b = b0 + (tid >> 1);
      float sum[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      if (b < nbins) {
        const float c = bins.centre[b];
        const int end = bins.start[b + 1];
        for (int i = bins.start[b] + (tid & 1); i < end; i += 2) {
          const float o = ((keys[i] - zmin) - c) * inv, o2 = o * o;
          sum[0] += 1.f; sum[1] += o; sum[2] += 0.5f * o2; sum[3] += o2 * o * (1.f / 6.f); sum[4] += o2 * o2 * (1.f / 24.f);
        }
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) sum[q] += __shfl_xor_sync(0xffffffffu, sum[q], 1);
      if (b < nbins && !(tid & 1)) {
#pragma unroll
        for (int q = 0; q < 5; ++q) bins.m[q][b] = sum[q];
      }
    }
    __syncthreads();
    // Taylor coefficients: e^(-(D + t - o)^2 / 2) = e^(-D^2 / 2) sum He_(n + m)(D) o^n / n! (-t)^m / m!; bins further than 6 widths
    // away do not count (1.5e-8 N).  A pair of lanes per bin, one for the bins below it and itself, one for those above.
    for (int b0 = 0; b0 < nbins; b0 += NT / 2) {
      const int b = b0 + (tid >> 1), dir = (tid & 1) ? 1 : -1;
      float l[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      if (b < nbins) {
        const float c = bins.centre[b];
        for (int j = dir > 0 ? b + 1 : b; j >= 0 && j < nbins; j += dir) {
          const float D = (c - bins.centre[j]) * inv;
          if (fabsf(D) > 6.f) break;
          float he[9];
          he[0] = ex2f(-0.7213475204f * D * D);
          he[1] = D * he[0];
#pragma unroll
          for (int q = 2; q < 9; ++q) he[q] = fmaf(D, he[q - 1], -float(q - 1) * he[q - 2]);
#pragma unroll
          for (int q = 0; q < 5; ++q) {
            const float m = bins.m[q][j];
#pragma unroll
            for (int r = 0; r < 5; ++r) l[r] = fmaf(he[q + r], m, l[r]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 5; ++r) l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
      if (b < nbins && !(tid & 1)) {
        bins.l[0][b] = l[0]; bins.l[1][b] = -l[1]; bins.l[2][b] = 0.5f * l[2]; bins.l[3][b] = l[3] * (-1.f / 6.f); bins.l[4][b] = l[4] * (1.f / 24.f);
      }
    }
    __syncthreads();
    float f[E], best = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = tid * E + e;
      f[e] = -1.f;
      if (i < n && !(i > 0 && v[e] == (e ? v[e > 0 ? e - 1 : 0] : keys[i - 1]))) {   // (else the same density as its predecessor)
        const int b = before + first[e] - 1;
        const float t = ((v[e] - zmin) - bins.centre[b]) * inv;
        f[e] = fmaf(t, fmaf(t, fmaf(t, fmaf(t, bins.l[4][b], bins.l[3][b]), bins.l[2][b]), bins.l[1][b]), bins.l[0][b]);
        best = fmaxf(best, f[e]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) wmax[warp] = best;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) best = fmaxf(best, wmax[w]);
    // What a value can be off by: the terms of order 5 left out on either side (|He_5 e^(-D^2/2)| < 6, 8^-5 / 120: 1.5e-6 N each), the
    // rounding of the offsets (1e-6 N), of the bins' sums (n 2^-24) and of the 45 x 5 products (together 7e-6 N): below 1.2e-5 N, twice for
    // two values compared.
    const float slack = 3e-5f * float(n);
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (f[e] >= 0.f && f[e] + slack >= best) list[atomicAdd(&count, 1)] = tid * E + e;
    __syncthreads();
    const int m = count;
    __shared__ double red_series[kSeries][NT / 32];
    float first_z = __int_as_float(0x7f800000), last_z = -first_z;
    for (int e = lane; e < m; e += 32) { const float x = keys[list[e]]; first_z = fminf(first_z, x); last_z = fmaxf(last_z, x); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      first_z = fminf(first_z, __shfl_xor_sync(0xffffffffu, first_z, o));
      last_z = fmaxf(last_z, __shfl_xor_sync(0xffffffffu, last_z, o));
    }
    const double middle = 0.5 * (double(first_z) + double(last_z));
    if (m == 1) {
      // nothing to tell apart
    } else if (m <= NT && (double(last_z) - middle) <= 0.125 * bw) {
      // The listed samples lie close together (around one mode): one pass over the samples gives the density about their middle in
      // fp64, e^(-(u - t)^2 / 2) = sum He_q(u) e^(-u^2 / 2) t^q / q!, and with it all their densities.  Left out with ten terms and
      // |t| <= 1/8: at most n 1.09 t^10 / sqrt(10!) = 5.4e-13 n (|He_q e^(-u^2/4)| < 1.09 sqrt(q!)); rounding adds less than 1e-13 n.
      const double inv = 1.0 / bw;
      double sum[kSeries] = {};
#pragma unroll 2
      for (int i = tid; i < n; i += NT) {
        const double u = (double(keys[i]) - middle) * inv;
        double h0 = exp_straight(-0.5 * u * u), h1 = u * h0;
        sum[0] += h0;
        sum[1] += h1;
#pragma unroll
        for (int q = 2; q < kSeries; ++q) {
          const double h2 = fma(u, h1, -double(q - 1) * h0);
          sum[q] += h2;
          h0 = h1;
          h1 = h2;
        }
      }
#pragma unroll
      for (int q = 0; q < kSeries; ++q) {
        const double w = warp_sum(sum[q]);
        if (lane == 0) red_series[q][warp] = w;
      }
      __syncthreads();
      if (tid < kSeries) {
        double all = 0.0;
        for (int w = 0; w < NT / 32; ++w) all += red_series[tid][w];
        red_series[tid][0] = all;
      }
      __syncthreads();
      double mine = -1.0;
      const int at = tid < m ? list[tid] : 0;
      if (tid < m) {
        const double t = (double(keys[at]) - middle) * inv;
        mine = red_series[kSeries - 1][0];
        for (int q = kSeries - 1; q > 0; --q) mine = fma(mine, t / double(q), red_series[q - 1][0]);
      }
      double top = mine;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
      if (lane == 0) bestv[warp] = top;
      __syncthreads();                                      // (count has been read, and the list)
      if (tid == 0) count = 0;
#pragma unroll
      for (int w = 0; w < NT / 32; ++w) top = fmax(top, bestv[w]);
      __syncthreads();
      if (tid < m && mine + 4e-12 * double(n) >= top) list[atomicAdd(&count, 1)] = at;
    } else {
    // sums of exponentials of the listed samples, two per warp at a time; eight terms at a time in fp32, those sums in fp64
    const float scale = float(0.8493218002880191 / bw);     // sqrt(log2(e) / 2) / width: e^(-u^2/2) = 2^-(scale (zk - zi))^2
    float* const dens = reinterpret_cast<float*>(list + n);
    float top = 0.f;
    for (int e = warp * 2; e < m; e += (NT / 32) * 2) {
      const float za = keys[list[e]], zb = keys[list[min(e + 1, m - 1)]];
      double fa = 0.0, fb = 0.0;
      for (int k0 = lane; k0 < n; k0 += 256) {
        float pa = 0.f, pb = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int k = k0 + 32 * q;
          if (k < n) {
            const float x = keys[k], ta = (x - za) * scale, tb = (x - zb) * scale;
            pa += ex2f(-ta * ta);
            pb += ex2f(-tb * tb);
          }
        }
        fa += double(pa);
        fb += double(pb);
      }
      fa = warp_sum(fa);
      fb = warp_sum(fb);
      if (lane == 0) { dens[e] = float(fa); if (e + 1 < m) dens[e + 1] = float(fb); }
      top = fmaxf(top, fmaxf(float(fa), float(fb)));
    }
    __syncthreads();                                        // (count and wmax have been read)
    if (tid == 0) count = 0;
    if (lane == 0) wmax[warp] = top;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) top = fmaxf(top, wmax[w]);
    // What these can be off by: the exponent (seven roundings) by 4.2e-7 of itself, which changes a term by at most 1.6e-7; the
    // exponential by 2^-22, the sums of eight terms and the last rounding by 10 2^-24 of the sum; twice for two values compared.
    const float slack2 = 3.2e-7f * float(n) + 1.8e-6f * top;
    int keep[(kMaxSearchSamples + NT - 1) / NT], nk = 0;
#pragma unroll
    for (int r = 0; r < (kMaxSearchSamples + NT - 1) / NT; ++r) {
      const int e = r * NT + tid;
      keep[r] = (e < m && dens[e] + slack2 >= top) ? list[e] : -1;
      nk += keep[r] >= 0;
    }
    __syncthreads();
    int at = nk ? atomicAdd(&count, nk) : 0;
#pragma unroll
    for (int r = 0; r < (kMaxSearchSamples + NT - 1) / NT; ++r)
      if (keep[r] >= 0) list[at++] = keep[r];
    }
  } else {
    for (int i = tid; i < n; i += NT) list[i] = i;
    if (tid == 0) count = n;
  }
  __syncthreads();
  // fp64 densities of what is left, one warp per sample
  const int m = count;
  const double inv64 = 1.0 / bw;
  double bv = -1.0;
  int bi = 0x7fffffff;
  for (int e = warp; e < m && m > 1; e += NT / 32) {
    const int i = list[e];
    const double zi = double(keys[i]);
    double dsum = 0.0;
    for (int k = lane; k < n; k += 32) { const double u = (double(keys[k]) - zi) * inv64; dsum += exp(-0.5 * u * u); }
    dsum = warp_sum(dsum);
    if (dsum > bv || (dsum == bv && i < bi)) { bv = dsum; bi = i; }
  }
  if (m == 1) bi = list[0];
  if (lane == 0) { bestv[warp] = bv; besti[warp] = bi; }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NT / 32; ++w)
    if (bestv[w] > bv || (bestv[w] == bv && besti[w] < bi)) { bv = bestv[w]; bi = besti[w]; }
  return bi;
}

// Mean squared residual of the least-squares line over the sorted samples i0 .. i1 - 1, as it is defined.  Where the errors that are
// compared are zero but for rounding (two distinct values inside, a straight stretch of the activation) the order of the additions
// decides, so it is a fixed one: 256 running sums, sample i0 + s + 256 k to sum s, added up in trees of 32, those in ascending order.
// By one warp:
__device__ __forceinline__ double residual_by_warp(const float* keys, const double* gs, int i0, int i1) {
  const int lane = threadIdx.x & 31, cnt = i1 - i0;
  if (cnt < 2) return 0.0;
  auto total = [&](auto term) {
    double t = 0.0;
    for (int s0 = 0; s0 < NT && s0 < cnt; s0 += 32) {        // (what is left out adds zeros)
      double sum = 0.0;
      for (int i = i0 + s0 + lane; i < i1; i += NT) sum += term(i);
      t += warp_sum(sum);
    }
    return t;
  };
  const double q = 1.0 / double(cnt);
  const double mz = total([&](int i) { return double(keys[i]); }) * q, mg = total([&](int i) { return gs[i]; }) * q;
  const double vzz = total([&](int i) { const double dz = double(keys[i]) - mz; return dz * dz; }) * q;
  if (!(vzz > 1e-30)) return 0.0;
  const double sl = total([&](int i) { return (double(keys[i]) - mz) * (gs[i] - mg); }) * q / vzz;
  return total([&](int i) { const double r = (gs[i] - mg) - sl * (double(keys[i]) - mz); return r * r; }) * q;
}
// By all threads, a tree of 32 per warp, for the two candidates of a step: whether the left one's is smaller.  What is found on the way stays
// in shared memory, because registers are what the walk has none left of.  (ReLU, where most steps of a wide range are undecided, 16384 x 2048:
// 26.3 -> 10.5 ms of steps of 0.005, 3.2 -> 1.9 of 0.05.)
struct Candidates {
  int from[2], to[2];                    // [left, right]
  double part[2][2][NT / 32];            // [side][sum][warp]
  double mz[2], mg[2], vzz[2], slope[2], err[2];
};
__device__ __forceinline__ bool left_is_smaller(const float* keys, const double* gs, Candidates& c) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll 1
  for (int stage = 0; stage < 3; ++stage) {                  // means; their second moments; residuals
#pragma unroll 1
    for (int e = 0; e < 4; ++e) {
      const int side = e >> 1, k = e & 1, to = c.to[side];
      double sum = 0.0;
      for (int i = c.from[side] + tid; i < to; i += NT) {
        double z = double(keys[i]), g = gs[i];
        if (stage > 0) { z -= c.mz[side]; g -= c.mg[side]; }
        if (stage == 0) sum += k ? g : z;
        else if (stage == 1) sum = fma(z, k ? g : z, sum);
        else { const double r = fma(-c.slope[side], z, g); sum = fma(r, r, sum); }
      }
      sum = warp_sum(sum);
      if (lane == 0) c.part[side][k][warp] = sum;
    }
    __syncthreads();
    if (tid < 2) {
      const int cnt = c.to[tid] - c.from[tid];
      const double q = 1.0 / double(cnt);
      double t[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        t[k] = 0.0;
        for (int w = 0; w < NT / 32 && w * 32 < cnt; ++w) t[k] += c.part[tid][k][w];
      }
      if (stage == 0) { c.mz[tid] = t[0] * q; c.mg[tid] = t[1] * q; }
      else if (stage == 1) { c.vzz[tid] = t[0] * q; c.slope[tid] = t[1] * q / (t[0] * q); }
      else c.err[tid] = cnt >= 2 && c.vzz[tid] > 1e-30 ? t[0] * q : 0.0;
    }
    __syncthreads();
  }
  return c.err[0] < c.err[1];
}

template <int E> __global__ void __launch_bounds__(NT, 4)
k_range_search(const float* __restrict__ z, long long ldz, const float* __restrict__ b1, int n,
               const float* __restrict__ thr, double t_all, double step, double n_root, int act, float* __restrict__ lo, float* __restrict__ hi,
               float* __restrict__ a, float* __restrict__ c, int* __restrict__ steps_out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* gs = reinterpret_cast<double*>(smem_raw);                // [NT E] activation of the sorted samples
  float* keys = reinterpret_cast<float*>(gs + NT * E);             // [NT E] sorted samples
  __shared__ double red[1][NT / 32];
  __shared__ float range_s[2];
  __shared__ union Scratch { Bins bins; Steps steps; __device__ Scratch() {} } scratch;
  __shared__ Ahead ahead;
  __shared__ Candidates candidates;
  __shared__ double base_m[5];                                     // moments of the range so far (the walk starts anew from time to time)
  __shared__ int base_k[2], base_end[2], total_steps, finished;
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  float v[E];
  load_samples<E>(v, z, ldz, b1, j, n);
  sort_samples<E>(v, keys);
#pragma unroll
  for (int e = 0; e < E; ++e) keys[tid * E + e] = v[e];
  // mean and standard deviation (N - 1 in the denominator) of the samples
  double s1[1] = {0.0}, s2[1] = {0.0};
#pragma unroll
  for (int e = 0; e < E; ++e) if (tid * E + e < n) s1[0] += double(v[e]);
  block_sums<1>(s1, red);
  const double mean = s1[0] / double(n);
#pragma unroll
  for (int e = 0; e < E; ++e) if (tid * E + e < n) { const double dz = double(v[e]) - mean; s2[0] += dz * dz; }
  block_sums<1>(s2, red);
  const double bw = n > 1 ? 1.06 * sqrt(s2[0] / double(n - 1)) * n_root : 0.0;     // (n_root: n^(-1/5))
  const int ic = bw > 0.0 ? densest_sample<E>(v, keys, n, bw, scratch.bins, reinterpret_cast<int*>(gs)) : 0;
  const double cen = double(keys[ic]);
  __syncthreads();                                                 // (the list in the place of gs has been read)
#pragma unroll
  for (int e = 0; e < E; ++e) gs[tid * E + e] = tid * E + e < n ? activation_f64(double(v[e]), act) : 0.0;
  __syncthreads();
  // number of samples below x
  auto lower = [&](double x) {
    int l = 0, r = n;
    while (l < r) { const int m = (l + r) >> 1; if (double(keys[m]) < x) l = m + 1; else r = m; }
    return l;
  };
  const double gc = gs[ic], zmin = double(keys[0]), zmax = double(keys[n - 1]);
  const double t = thr ? double(thr[j]) : t_all;
  const int cap = 4 + 2 * int(fmin(1.0e7, (zmax - zmin) / step + 2.0));   // the loop ends long before; a guard against a bad step
  Steps& st = scratch.steps;
  if (tid < 5) base_m[tid] = 0.0;
  if (tid == 0) {
    base_k[0] = base_k[1] = total_steps = finished = 0;
    base_end[0] = base_end[1] = lower(cen);                        // samples inside: none yet
  }
  do {
    __syncthreads();                                               // (the bins, or the steps before, have been read)
    // (1) where the next kMaxSteps steps on either side end, (2) what each adds about the centroid (y = z - centroid, g = activation -
    // activation at the centroid; sums of y, g, y y, y g, g g), (3) running sums
    if (tid < 2) st.end[tid][0] = base_end[tid];
    for (int e = tid; e < 2 * kMaxSteps; e += NT) {
      const int side = e & 1, k = (e >> 1) + 1;
      st.end[side][k] = lower(side ? cen + (base_k[1] + k) * step : cen - (base_k[0] + k) * step);
    }
    __syncthreads();
    for (int e = tid; e < 2 * kMaxSteps; e += NT) {
      const int side = e & 1, k = e >> 1;
      const int p0 = side ? st.end[1][k] : st.end[0][k + 1], p1 = side ? st.end[1][k + 1] : st.end[0][k];
      double m0 = 0.0, m1 = 0.0, m2 = 0.0, m3 = 0.0, m4 = 0.0;
      for (int i = p0; i < p1; ++i) {
        const double y = double(keys[i]) - cen, q = gs[i] - gc;
        m0 += y; m1 += q; m2 += y * y; m3 += y * q; m4 += q * q;
      }
      st.m[side][0][k + 1] = m0; st.m[side][1][k + 1] = m1; st.m[side][2][k + 1] = m2; st.m[side][3][k + 1] = m3; st.m[side][4][k + 1] = m4;
    }
    __syncthreads();
    for (int q = tid >> 5; q < 10; q += NT / 32) {
      double* const m = st.m[q & 1][q >> 1];
      double carry = 0.0;
      if (lane == 0) m[0] = 0.0;
      for (int k0 = 1; k0 <= kMaxSteps; k0 += 32) {                // (kMaxSteps is a multiple of 32)
        double x = m[k0 + lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const double up = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += up; }
        x += carry;
        m[k0 + lane] = x;
        carry = __shfl_sync(0xffffffffu, x, 31);
      }
    }
    __syncthreads();
    // Range after i steps to the left and jr to the right, i + jr <= kAhead: number s (s + 1) / 2 + jr, s = i + jr, and a thread's.  (What
    // follows is the same for all threads: kl, kr, nsteps, done.)
    int s_mine = 0;
    while ((s_mine + 1) * (s_mine + 2) / 2 <= tid) ++s_mine;
    const int j_mine = min(tid - s_mine * (s_mine + 1) / 2, kAhead), i_mine = max(0, min(s_mine, kAhead) - j_mine);
    int kl = 0, kr = 0, nsteps = total_steps;
    bool done = false;
    while (!done && kl + kAhead <= kMaxSteps && kr + kAhead <= kMaxSteps) {
      // the thread's range: error from the moments (times its number of samples, and so on, to have one reciprocal), and what it can be
      // off by (infinite where the moments cancel)
      const int e0 = st.end[0][kl + i_mine], e1 = st.end[1][kr + j_mine], cnt = e1 - e0;
      {
        bool zero = cnt < 2;
        if (act == TARDIS_ACT_RELU) zero = zero || keys[min(e0, n - 1)] > 0.f || keys[max(e1 - 1, 0)] <= 0.f;   // (one straight piece: exactly zero)
        double m[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) m[q] = base_m[q] + (st.m[0][q][kl + i_mine] + st.m[1][q][kr + j_mine]);
        const double q = double(cnt), yy = m[2] * q, gg = m[4] * q;
        const double vyy = yy - m[0] * m[0], vyg = m[3] * q - m[0] * m[1], vgg = gg - m[1] * m[1];
        // Every moment is off by less than c = (n + 20) 2^-53 = 2.3e-13 of the sum of its terms' sizes (n additions, a few roundings
        // in a term and in joining the parts), and |yg| <= sqrt(yy gg): vyy by 3 c yy, vyg by 3 c sqrt(yy gg), vgg by 3 c gg, so
        // err q^2 by 3 c gg (1 + sqrt(yy / vyy))^2 <= 7e-13 gg k^2.
        const float k = 1.f + __fdividef(float(yy), float(vyy)), iq = __fdividef(1.f, float(q));
        const bool cancels = !(vyy > 1e-8 * yy && vyy > 1e-25 * q * q);
        ahead.off[tid] = zero ? 0.f : (cancels ? __int_as_float(0x7f800000) : fmaxf(1e-12f * float(gg) * iq * iq * k * k, 1e-37f));
        // (vgg vyy - vyg^2) / (vyy q^2), the reciprocal by two Newton steps from the 20 bits of an approximate one
        const double den = cancels ? 1.0 : vyy * q * q;
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(den));
        y = fma(y, fma(-den, y, 1.0), y);
        y = fma(y, fma(-den, y, 1.0), y);
        ahead.err[tid] = zero || cancels ? 0.0 : (vgg * vyy - vyg * vyg) * y;
      }
      __syncthreads();
      // what would be done from the range: 0 right, 1 left, 2 nothing (enough samples inside), 3 the errors do not tell; and the range that
      // follows (the same one where the walk has to stop)
      {
        const double l = cen - (base_k[0] + kl + i_mine) * step, u = cen + (base_k[1] + kr + j_mine) * step;
        const int to_left = min(tid + s_mine + 1, NT - 1), to_right = min(tid + s_mine + 2, NT - 1);   // (of the last ones: never used)
        const double el = ahead.err[to_left], er = ahead.err[to_right];
        const float o = ahead.off[to_left] + ahead.off[to_right];
        int move = !(fabs(el - er) > double(o)) && o != 0.f ? 3 : (el < er ? 1 : 0);
        if (l <= zmin) move = 0;
        if (u > zmax) move = 1;                                    // (not both sides: every sample would be inside)
        if (double(cnt) >= t * double(n) || cnt == n || nsteps + s_mine >= cap) move = 2;
        ahead.next[tid] = uint16_t((s_mine >= kAhead || move >= 2 ? tid : (move == 1 ? to_left : to_right)) | move << 8 | s_mine << 10);
      }
      __syncthreads();
      int last = 0, at = ahead.next[0];
      while ((at & 0xff) != last) { last = at & 0xff; at = ahead.next[last]; }
      const int what = at >> 8 & 3, s_last = at >> 10;
      int jr = last - s_last * (s_last + 1) / 2, i = s_last - jr;
      if (s_last < kAhead) {
        done = what == 2;
        if (what == 3) {                                           // (every thread finds the same)
          const int l0 = st.end[0][kl + i + 1], p0 = st.end[0][kl + i], p1 = st.end[1][kr + jr], r1 = st.end[1][kr + jr + 1];
          bool left;
          if (r1 - l0 <= 64) {                                     // every warp for itself: no barriers (64 samples: 4.6 ms, 5.5 with them)
            left = residual_by_warp(keys, gs, l0, p1) < residual_by_warp(keys, gs, p0, r1);
          } else {
            if (tid == 0) { candidates.from[0] = l0; candidates.to[0] = p1; candidates.from[1] = p0; candidates.to[1] = r1; }
            __syncthreads();
            left = left_is_smaller(keys, gs, candidates);
          }
          if (left) ++i; else ++jr;
        }
      }
      nsteps += i + jr;
      kl += i;
      kr += jr;
    }
    __syncthreads();                                               // (the sums so far have been read)
    if (tid < 5) base_m[tid] += st.m[0][tid][kl] + st.m[1][tid][kr];
    if (tid == 0) {
      base_k[0] += kl; base_k[1] += kr;
      base_end[0] = st.end[0][kl]; base_end[1] = st.end[1][kr];
      total_steps = nsteps;
      finished = done;
    }
    __syncthreads();
  } while (!finished);
  if (tid == 0) {
    range_s[0] = float(cen - base_k[0] * step);
    range_s[1] = float(cen + base_k[1] * step);
    if (steps_out) steps_out[j] = total_steps;
  }
  __syncthreads();
  double g[E];
#pragma unroll
  for (int e = 0; e < E; ++e) { v[e] = keys[e * NT + tid]; g[e] = gs[e * NT + tid]; }
  fit_and_store<E>(v, g, range_s[0], range_s[1], act, j, lo, hi, a, c);
}

// Error contribution of every neuron (Section 5.1.1, the E of the neuron-level thresholds): the mean squared residual of
// the least-squares line over the neuron's samples inside its range [lo_j, hi_j), as Algorithm 1's approx_error measures it.
// (The samples inside are told by comparison: no order is needed.)
template <int E> __global__ void __launch_bounds__(NT)
k_neuron_error(const float* __restrict__ z, long long ldz, const float* __restrict__ b1, int n, int act,
               const float* __restrict__ lo, const float* __restrict__ hi, float* __restrict__ err) {
  __shared__ double red3[3][NT / 32];
  __shared__ double red2[2][NT / 32];
  __shared__ double red1[1][NT / 32];
  const int j = blockIdx.x;
  const double l = double(lo[j]), u = double(hi[j]);
  float v[E];
  double g[E];
  load_samples<E>(v, z, ldz, b1, j, n);
  double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const double x = double(v[e]);
    const bool in = e * NT + threadIdx.x < n && x >= l && x < u;
    g[e] = in ? activation_f64(x, act) : 0.0;
    if (in) { s[0] += 1.0; s[1] += x; s[2] += g[e]; }
    else v[e] = __int_as_float(0x7f800000);
  }
  block_sums<3>(s, red3);
  double r = 0.0;
  if (s[0] >= 2.0) {                                        // (uniform over the CTA)
    const double q = 1.0 / s[0], mz = s[1] * q, mg = s[2] * q;
    double m[2] = {0.0, 0.0};
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (v[e] < __int_as_float(0x7f800000)) { const double dz = double(v[e]) - mz; m[0] += dz * dz; m[1] += dz * (g[e] - mg); }
    block_sums<2>(m, red2);
    const double vzz = m[0] * q;
    if (vzz > 1e-30) {
      const double sl = m[1] * q / vzz;
      double rr[1] = {0.0};
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (v[e] < __int_as_float(0x7f800000)) { const double w = (g[e] - mg) - sl * (double(v[e]) - mz); rr[0] += w * w; }
      block_sums<1>(rr, red1);
      r = rr[0] * q;
    }
  }
  if (threadIdx.x == 0) err[j] = float(r);
}

// Neuron-level thresholds (Section 5.1.1): minimise sum_j E_j t_j subject to sum_j t_j = t_layer h, read with the box
// t_min <= t_j <= t_max.  A linear objective over a box with one equality: every neuron starts at t_min and the budget
// (t_layer - t_min) h goes, t_max - t_min each, to the neurons in order of increasing error (the smaller index first among
// equals).  Eight lanes find a neuron's place in that order by counting an eighth of the errors each (a thread per neuron
// leaves more than half of the SMs idle at 16384 neurons: 85 us), then it takes its share of what is left for it.
__global__ void __launch_bounds__(NT)
k_neuron_thresholds(const float* __restrict__ err, int h, double t_layer, double t_min, double t_max, float* __restrict__ t) {
  __shared__ __align__(16) float tile[NT * 4];
  const int j = blockIdx.x * (NT / 8) + (threadIdx.x >> 3), part = threadIdx.x & 7;
  const float ej = j < h ? err[j] : 0.f;
  int rank = 0;
  for (int base = 0; base < h; base += NT * 4) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = base + r * NT + threadIdx.x;
      tile[r * NT + threadIdx.x] = i < h ? err[i] : __int_as_float(0x7f800000);
    }
    __syncthreads();
    // equal errors count where their neuron comes first: in a tile that lies in front of the CTA's neurons or behind them the same for all
    const float4* const at = reinterpret_cast<const float4*>(tile);
    if (base + NT * 4 <= int(blockIdx.x) * (NT / 8)) {
#pragma unroll 8
      for (int i = part; i < NT; i += 8) { const float4 v = at[i]; rank += (v.x <= ej) + (v.y <= ej) + (v.z <= ej) + (v.w <= ej); }
    } else if (base >= (int(blockIdx.x) + 1) * (NT / 8)) {
#pragma unroll 8
      for (int i = part; i < NT; i += 8) { const float4 v = at[i]; rank += (v.x < ej) + (v.y < ej) + (v.z < ej) + (v.w < ej); }
    } else {
#pragma unroll 8
      for (int i = part; i < NT * 4; i += 8) {
        const float v = tile[i];
        rank += (v < ej || (v == ej && base + i < j)) ? 1 : 0;
      }
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
  if (j >= h || part) return;
  const double cap = t_max - t_min, budget = (t_layer - t_min) * double(h);
  const double give = fmin(cap, fmax(0.0, budget - double(rank) * cap));
  t[j] = float(t_min + give);
}

// Calls f with the number of samples per thread (a power of two up to MOST) that covers n samples, as a compile-time constant
template <int MOST, int E = 1, typename F> static tardis_status_t with_samples(int n, F&& f) {
  if constexpr (E > MOST) { (void)n; (void)f; return TARDIS_ERR_UNSUPPORTED; }
  else return n <= NT * E ? f(std::integral_constant<int, E>()) : with_samples<MOST, E * 2>(n, static_cast<F&&>(f));
}

}  // namespace cal

tardis_status_t launch_neuron_thresholds(int h, int n, const float* z, long long ldz, const float* b1, const float* lo, const float* hi,
                                         int act, double t_layer, double t_min, double t_max, float* err, float* t, cudaStream_t s) {
  if (n < 1 || n > cal::kMaxSearchSamples) return TARDIS_ERR_UNSUPPORTED;
  const tardis_status_t st = cal::with_samples<cal::kMaxSearchSamples / cal::NT>(n, [&](auto e) {
    cal::k_neuron_error<decltype(e)::value><<<h, cal::NT, 0, s>>>(z, ldz, b1, n, act, lo, hi, err);
    TARDIS_CUDA_TRY(cudaGetLastError());
    return TARDIS_OK;
  });
  if (st != TARDIS_OK) return st;
  cal::k_neuron_thresholds<<<(h * 8 + cal::NT - 1) / cal::NT, cal::NT, 0, s>>>(err, h, t_layer, t_min, t_max, t);
  TARDIS_CUDA_TRY(cudaGetLastError());
  return TARDIS_OK;
}

tardis_status_t launch_calibrate(int h, int n, const float* z, long long ldz, const float* b1, double q_lo, double q_hi, int act,
                                 float* lo, float* hi, float* a, float* c, cudaStream_t s) {
  if (n < 1 || n > cal::kMaxSamples) return TARDIS_ERR_UNSUPPORTED;
  return cal::with_samples<cal::kMaxSamples / cal::NT>(n, [&](auto e) {
    constexpr int E = decltype(e)::value;
    const auto kernel = act == TARDIS_ACT_GELU_ERF ? cal::k_calibrate<E, true> : cal::k_calibrate<E, false>;
    kernel<<<h, cal::NT, size_t(cal::NT) * E * sizeof(float), s>>>(z, ldz, b1, n, q_lo, q_hi, act, lo, hi, a, c);
    TARDIS_CUDA_TRY(cudaGetLastError());
    return TARDIS_OK;
  });
}

tardis_status_t launch_range_search(int h, int n, const float* z, long long ldz, const float* b1, const float* thr, double t_all,
                                    double step, int act, float* lo, float* hi, float* a, float* c, int* steps_out, cudaStream_t s) {
  if (n < 1 || n > cal::kMaxSearchSamples) return TARDIS_ERR_UNSUPPORTED;
  return cal::with_samples<cal::kMaxSearchSamples / cal::NT>(n, [&](auto e) {
    constexpr int E = decltype(e)::value;
    cal::k_range_search<E><<<h, cal::NT, size_t(cal::NT) * E * (sizeof(double) + sizeof(float)), s>>>(z, ldz, b1, n, thr, t_all, step, pow(double(n), -0.2), act,
                                                                                                     lo, hi, a, c, steps_out);
    TARDIS_CUDA_TRY(cudaGetLastError());
    return TARDIS_OK;
  });
}

}  // namespace tardis
