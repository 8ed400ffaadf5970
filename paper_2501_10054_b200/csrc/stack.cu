// A chain of partially linear FFN layers on one residual stream: per layer an optional layer normalisation of the
// stream, the layer's forward (tardis_ffn_forward, whatever path it picks), and the addition of its output to the
// stream.  The paper has no counterpart of this call (it replaces the FFN block inside an existing model, Section 6);
// it is the shape in which a decoder hands the FFN blocks of consecutive layers to this library, without attention.
//
// Two small kernels live here.  k_update_norm (one CTA per token, the row in registers, fp32) adds the previous layer's
// output to the stream and normalises the result for the next layer in one pass; k_stream_update adds the last layer's
// output.  Both take part in the programmatic hand-over between launches: they let the next launch start at once
// (the fused decode kernel then loads its predictor blocks while the row is being normalised) and wait for the launch
// before them only where they first touch its results.  Everything else is the per-layer forward.  Layers that are one launch of the
// fused kernel (one or two tokens, four on narrow layers) need neither: see FusedChain.
#include "common.cuh"

namespace tardis {
namespace {

constexpr int LN_THREADS = 512;
constexpr int LN_MAXVEC = 3;    // vectors of 8 elements per thread: d_model up to 12288

__device__ __forceinline__ float block_sum(float v, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();                       // (sh may still be read from the previous sum)
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  v = sh[lane & (LN_THREADS / 32 - 1)];  // every warp adds the same numbers in the same order
#pragma unroll
  for (int o = LN_THREADS / 64; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 8 consecutive elements (16-byte aligned) as fp32, and back
__device__ __forceinline__ void load8(float (&v)[8], const float* p) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(float (&v)[8], const __nv_bfloat16* p) {
  const uint4 a = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}
__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&v)[8]) {
  __nv_bfloat162 o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
  *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(o);
}
// 8 consecutive values of a table of the caller's, which need not begin on a 16-byte boundary
__device__ __forceinline__ void load_table(float (&v)[8], const float* p) {
  if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) return load8(v, p);
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = p[q];
}
// v = residual ? v + f : f, rounded as it is stored
template <typename T> __device__ __forceinline__ void add_output(float (&v)[8], const float (&f)[8], int residual) {
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = residual ? to_f32<T>(from_f32<T>(v[i] + f[i])) : f[i];
}

// stream[t][:] = src[t][:] (the stream itself, or x for the first layer that needs it), with the previous layer's output f[t][:]
// (update: added when `residual`, else in its place), then
// out[t][i] = (stream[t][i] - mean_t) / sqrt(var_t + eps) * gamma[i] + beta[i]; mean and variance (1/d, not 1/(d-1)) over the
// row; without `normalise` out is the stream itself.  One CTA per token, the row in registers: bound by the latency of one load, two
// sums and one store (4096 elements, one token: 16 us with an element per load and 48 guarded steps for any d_model, 3 us now).
template <typename T, int NV>
__global__ void __launch_bounds__(LN_THREADS) k_update_norm(const T* src, T* stream, const T* __restrict__ f, int update, int residual,
                                                            int normalise, T* __restrict__ out, const float* gamma, const float* beta, int d,
                                                            float eps) {
  __shared__ float sh[LN_THREADS / 32];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // gamma and beta may be written by a launch of the caller's that is still running: asked into L2 now, read behind the wait (read from
  // memory behind it: 0.8 us more per layer)
  for (int i = threadIdx.x * 32; i < d && normalise; i += LN_THREADS * 32) {
    if (gamma) asm volatile("prefetch.global.L2 [%0];" ::"l"(gamma + i));
    if (beta) asm volatile("prefetch.global.L2 [%0];" ::"l"(beta + i));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");          // the launch before wrote f (or the stream)
  const size_t row = size_t(blockIdx.x) * d;
  float v[NV][8], w[NV][8], ga[NV][8], be[NV][8];
#pragma unroll
  for (int e = 0; e < NV; ++e) {                               // (d is a multiple of 8)
    const int i = (threadIdx.x + e * LN_THREADS) * 8;
#pragma unroll
    for (int q = 0; q < 8; ++q) { v[e][q] = 0.f; ga[e][q] = 1.f; be[e][q] = 0.f; }
    if (i < d) {
      load8(v[e], src + row + i);
      if (update) load8(w[e], f + row + i);
    }
  }
#pragma unroll
  for (int e = 0; e < NV; ++e) {                               // (behind the row's loads: these arrive while the row is summed up)
    const int i = (threadIdx.x + e * LN_THREADS) * 8;
    if (normalise && i < d) {
      if (gamma) load_table(ga[e], gamma + i);
      if (beta) load_table(be[e], beta + i);
    }
  }
  float s = 0.f;
#pragma unroll
  for (int e = 0; e < NV; ++e) {
    const int i = (threadIdx.x + e * LN_THREADS) * 8;
    if (i < d) {
      if (update) add_output<T>(v[e], w[e], residual);
      if (update || src != stream) store8(stream + row + i, v[e]);
#pragma unroll
      for (int q = 0; q < 8; ++q) s += v[e][q];
    }
  }
  if (normalise) {
    const float mean = block_sum(s, sh) / float(d);
    float sq = 0.f;
#pragma unroll
    for (int e = 0; e < NV; ++e)
      if ((threadIdx.x + e * LN_THREADS) * 8 < d) {
#pragma unroll
        for (int q = 0; q < 8; ++q) { const float c = v[e][q] - mean; sq += c * c; }
      }
    const float rstd = rsqrtf(block_sum(sq, sh) / float(d) + eps);
#pragma unroll
    for (int e = 0; e < NV; ++e)
#pragma unroll
      for (int q = 0; q < 8; ++q) v[e][q] = (v[e][q] - mean) * rstd * ga[e][q] + be[e][q];
  }
#pragma unroll
  for (int e = 0; e < NV; ++e) {
    const int i = (threadIdx.x + e * LN_THREADS) * 8;
    if (i < d) store8(out + row + i, v[e]);
  }
}

// stream = src + f (residual) or stream = f: after the last layer
template <typename T>
__global__ void __launch_bounds__(128) k_stream_update(const T* src, T* stream, const T* __restrict__ f, size_t count, int residual) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (size_t i = (size_t(blockIdx.x) * blockDim.x + threadIdx.x) * 8; i < count; i += size_t(gridDim.x) * blockDim.x * 8) {
    float v[8], w[8];
    load8(v, src + i);
    load8(w, f + i);
    add_output<T>(v, w, residual);
    store8(stream + i, v);
  }
}

template <typename... Args>
cudaError_t launch_chained(void (*kernel)(Args...), dim3 grid, dim3 block, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = 0; cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T>
tardis_status_t run_stack(const tardis_stack_desc_t* desc, const void* x, void* y, void* work, void* keep, int64_t n, cudaStream_t s) {
  Handle* H0 = reinterpret_cast<Handle*>(desc->layers[0]);
  const int d = H0->d;
  const size_t count = size_t(n) * d;
  T* stream = static_cast<T*>(y);
  const T* src = static_cast<const T*>(x);                     // where the stream's values are: in x until a kernel has written y
  const int norm = desc->normalise != 0 ? 1 : 0;
  const auto update_norm = d <= LN_THREADS * 8 ? k_update_norm<T, 1> : (d <= LN_THREADS * 16 ? k_update_norm<T, 2> : k_update_norm<T, LN_MAXVEC>);
  T* fprev = nullptr;                                          // the output that is still to be added to the stream
  auto add_last = [&](const T* f) -> tardis_status_t {
    const size_t blocks = (count / 8 + 127) / 128;
    TARDIS_CUDA_TRY(launch_chained(k_stream_update<T>, dim3(unsigned(blocks < 4096 ? blocks : 4096)), dim3(128), s, src, stream, f, count, int(desc->residual)));
    src = stream;
    return TARDIS_OK;
  };
  for (int l = 0; l < desc->n_layers; ++l) {
    // with `keep`, the layer's input and output stay where the caller can read them; else two buffers for the inputs take
    // turns with one for the output (the update of layer l + 1 reads the output of layer l while writing its own input)
    T* xin = keep ? static_cast<T*>(keep) + size_t(2 * l) * count : static_cast<T*>(work);
    T* fout = keep ? static_cast<T*>(keep) + size_t(2 * l + 1) * count : static_cast<T*>(work) + count;
    const T* layer_in = src;
    Handle* const H = reinterpret_cast<Handle*>(desc->layers[l]);
    if (fused_chain_serves(H, n)) {
      // One launch for the layer: the kernel normalises the stream as it reads it and its last CTA adds the output (4 layers of
      // 4096/16384, one token: 98.3 us against 104.6 with the small kernels between the layers)
      if (fprev) { const tardis_status_t st = add_last(fprev); if (st != TARDIS_OK) return st; }
      FusedChain c = {};
      c.normalise = norm != 0; c.residual = desc->residual != 0; c.eps = desc->ln_eps;
      c.gamma = norm && desc->ln_gamma ? desc->ln_gamma[l] : nullptr; c.beta = norm && desc->ln_beta ? desc->ln_beta[l] : nullptr;
      c.keep_in = keep ? reinterpret_cast<__nv_bfloat16*>(xin) : nullptr; c.keep_out = keep ? reinterpret_cast<__nv_bfloat16*>(fout) : nullptr;
      H->last_stream = s;
      const tardis_status_t st = launch_fused_forward(H, src, stream, int(n), s, &c);
      if (st != TARDIS_OK) return st;
      H->last_path = 2; H->calls += 1; H->tokens += uint64_t(n);
      src = stream;
      fprev = nullptr;
      continue;
    }
    if (norm || keep || l > 0) {
      TARDIS_CUDA_TRY(launch_chained(update_norm, dim3(unsigned(n)), dim3(LN_THREADS), s, src, stream, static_cast<const T*>(fprev ? fprev : stream),
                                     fprev ? 1 : 0, int(desc->residual), norm, xin, norm && desc->ln_gamma ? desc->ln_gamma[l] : static_cast<const float*>(nullptr),
                                     norm && desc->ln_beta ? desc->ln_beta[l] : static_cast<const float*>(nullptr), d, desc->ln_eps));
      layer_in = xin;
      src = stream;
    }
    const tardis_status_t st = tardis_ffn_forward(desc->layers[l], layer_in, fout, n, reinterpret_cast<tardis_stream_t>(s));
    if (st != TARDIS_OK) return st;
    fprev = fout;
  }
  return fprev ? add_last(fprev) : TARDIS_OK;
}

}  // namespace

tardis_status_t launch_stack_forward(const tardis_stack_desc_t* desc, const void* x, void* y, void* work, void* keep, int64_t n,
                                     cudaStream_t s) {
  Handle* H0 = reinterpret_cast<Handle*>(desc->layers[0]);
  if (H0->d > LN_THREADS * 8 * LN_MAXVEC) return TARDIS_ERR_UNSUPPORTED;
  return H0->dtype == TARDIS_F32 ? run_stack<float>(desc, x, y, work, keep, n, s) : run_stack<__nv_bfloat16>(desc, x, y, work, keep, n, s);
}

}  // namespace tardis
