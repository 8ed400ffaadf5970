// Shared declarations of libtardis (internal; the public interface is include/tardis.h).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tardis.h"

namespace tardis {

constexpr uint64_t kMagic = 0x7A2D15F01DULL;
constexpr int kGenericChunk = 256;   // tokens per pass of the generic kernels (scratch is sized for this)
constexpr int kDecodeMaxTokens = 16; // largest batch the fused decode kernel takes (4 tokens per launch) on layers of up to 4096
                                     // channels; 13 on wider ones (measured against the batched path, see fused_max_tokens)
constexpr int kStaticMaxTokens = 64; // largest batch of the forward that keeps its scratch in the library image

// device counter slots
enum { CTR_FLAGGED_TOTAL = 0, CTR_FLAGGED_MAX = 1, CTR_ERROR = 2, CTR_RECHECKS = 3, CTR_TICKET = 4, CTR_LAST_UNION = 5, CTR_COUNT = 8 };

struct Handle {
  uint64_t magic;
  int d, h, dtype, act, G, ngroups;
  int bits;              // bits per predictor code (2, 4 or 8)
  size_t esize;
  int device;
  // state (device)
  void* W1;        // [h, d]   original rows (result fixing recomputes z_j from these)
  void* W2T;       // [h, d]   W2 transposed: row j = output weights of neuron j
  void* C;         // [d, d]   C[k, i] = W_f[i, k]  (the paper's folded matrix, row k = input channel k)
  float* bf;       // [d]
  float *lo, *hi, *a, *c, *b1;   // [h]; b1 is zeros when the layer has no bias
  uint32_t* codes; // [h, d/16]
  void* scale;     // [h, d/G]
  uint8_t* zero;   // [h, d/G]
  // fused-decode state (bf16 only; null otherwise)
  uint32_t* codes_mma;   // predictor codes re-packed into tensor-core fragment order
  float2* pmeta;         // [h/16 tiles][ngroups][16 rows] (scale, scale*zero)
  // scratch (device)
  float* yacc;           // [kGenericChunk, d] fp32 accumulator
  uint32_t* bitmap;      // [kGenericChunk, h/32]
  unsigned long long* counters;  // [CTR_COUNT]
  void* fscratch;        // fused decode state for calls of 1..4 tokens per launch (see fused.cu); null when not built
  int fused_max_tokens;  // calls of up to this many tokens go to that kernel when the path is chosen automatically
  void* dscratch;        // fused decode scratch (see decode.cu)
  size_t dscratch_bytes;
  void* bstate;          // batched / prefill state and scratch (see batched.cu); null when not built
  void* f32;             // state of the kernels for fp32 layers (see f32.cu); null for other layers
  void* few;             // state of the kernels for a few to 128 tokens (see few.cu); null when not built
  // debug capture (caller-owned)
  uint32_t* dbg_bitmap;
  double* dbg_scores;
  // host-side bookkeeping
  uint64_t calls, tokens, last_path, launches;
  cudaStream_t last_stream;
  int path_override;
  bool deterministic;    // y must not depend on the order in which partial sums arrive (tardis_set_deterministic)
  size_t bytes_folded, bytes_predictor, bytes_tables, bytes_w1, bytes_w2t, bytes_scratch;
  int num_sms;
};

void set_last_error(cudaError_t e, const char* where);

// Every device allocation of the library goes through here: cudaMalloc, or the failure that tardis_debug_fail_alloc
// has asked for (so that the clean-up after a failed allocation can be tested without exhausting a GPU).  The memory
// handed out sits between two guard areas that tardis_stats checks.
cudaError_t dev_malloc_raw(void** p, size_t bytes);
template <typename T> inline cudaError_t dev_malloc(T** p, size_t bytes) { return dev_malloc_raw(reinterpret_cast<void**>(p), bytes); }
void dev_free(void* p);   // what dev_malloc gave (null is fine)
size_t dev_room(size_t bytes);      // what an allocation takes of a block, guards included
void dev_reserve(size_t bytes);     // one block for the allocations that the running entry point is going to make (the sum of their dev_room)

#define TARDIS_CUDA_TRY(expr)                                  \
  do {                                                         \
    cudaError_t e__ = (expr);                                  \
    if (e__ != cudaSuccess) {                                  \
      ::tardis::set_last_error(e__, #expr);                    \
      return TARDIS_ERR_CUDA;                                  \
    }                                                          \
  } while (0)

// ---- kernels' host launchers (each returns after enqueueing on `s`) ----
tardis_status_t launch_fold(Handle* H, const tardis_fold_desc_t* desc, cudaStream_t s, bool skip_product = false);
tardis_status_t launch_fold_product(Handle* H, cudaStream_t s);   // the SIMT product alone
tardis_status_t launch_export_folded(Handle* H, void* Wf, float* bf, cudaStream_t s);
cudaError_t launch_transpose(const __nv_bfloat16* in, __nv_bfloat16* out, int rows, int cols, cudaStream_t s);   // out[cols, rows] from in[rows, cols]
tardis_status_t launch_generic_forward(Handle* H, const void* x, void* y, int64_t n, cudaStream_t s);
tardis_status_t launch_static_forward(Handle* H, const void* x, void* y, int64_t n, cudaStream_t s);
tardis_status_t decode_prepare(Handle* H, cudaStream_t s);                 // builds codes_mma, pmeta, scratch
tardis_status_t launch_decode_forward(Handle* H, const void* x, void* y, int n, cudaStream_t s);
void decode_release(Handle* H);
tardis_status_t decode_read_stamps(long long* out, int max_ctas);
size_t fused_room(const Handle* H);                                        // what fused_prepare or decode_prepare will allocate
tardis_status_t fused_prepare(Handle* H, cudaStream_t s);                  // builds the state of fused.cu (bf16, d_model <= 4608)
// A layer of a chain in one launch of the fused kernel: x is the residual stream s, the layer's input u is its normalisation (or s), and
// with f the layer's output y becomes s + f (residual) or f; y may be x.  keep_in, keep_out: null, or where u and f go.
struct FusedChain {
  bool normalise, residual;
  float eps;
  const float *gamma, *beta;                                                  // null: ones and zeros
  __nv_bfloat16 *keep_in, *keep_out;
};
tardis_status_t launch_fused_forward(Handle* H, const void* x, void* y, int n, cudaStream_t s, const FusedChain* chain = nullptr);
// Most tokens of a chain's layer that is one launch of the fused kernel.  Of the calls that tardis_ffn_forward gives to it as one launch those of
// three and four tokens only on narrow layers: every CTA normalises all tokens, which there takes less than the small kernels between the
// layers and wider less and less (three layers, us with the small kernels / inside: 2 tokens of 1024/4096 47.3 / 43.0, of 4544/18176 114.6 / 111.6; 4
// tokens of 1024/4096 56.9 / 56.2, of 2048/8192 73.7 / 74.9, of 4544/18176 152 / 159).
inline int max_chain_tokens(int d) { return d <= 1024 ? 4 : 2; }
bool fused_chain_serves(const Handle* H, int64_t n);
void fused_release(Handle* H);
tardis_status_t fused_set_deterministic(Handle* H, bool on);               // allocates the partial-output buffer of the mode
tardis_status_t fused_read_stamps(long long* out, int max_ctas);
tardis_status_t launch_wait_that_runs_out(Handle* H, long long limit_cycles, cudaStream_t s);   // UNSUPPORTED unless built with TARDIS_PHASE_STAMPS
size_t batched_room(const Handle* H);                                                         // what batched_prepare (and few_prepare) will allocate
tardis_status_t batched_prepare(Handle* H);                                                   // bf16 only: allocations
tardis_status_t batched_finish(Handle* H, const void* W2, cudaStream_t s);   // fills the batched state (W2 null: from W2T)
tardis_status_t launch_batched_forward(Handle* H, const void* x, void* y, int64_t n, cudaStream_t s);
void batched_release(Handle* H);
size_t few_room(const Handle* H);
tardis_status_t few_prepare(Handle* H);                                       // few.cu: allocations
tardis_status_t few_finish(Handle* H, const void* W2, const void* Wf, cudaStream_t s);   // fills its state (W2 [d, h], W_f [d, d] row-major)
tardis_status_t launch_few_forward(Handle* H, const void* x, void* y, int n, const float* smaxrow, cudaStream_t s);
void few_release(Handle* H);
size_t f32_room(const Handle* H);
tardis_status_t f32_prepare(Handle* H, cudaStream_t s);                        // f32.cu (fp32 layers only)
tardis_status_t launch_f32_forward(Handle* H, const void* x, void* y, int64_t n, cudaStream_t s);
void f32_release(Handle* H);
tardis_status_t launch_stack_forward(const tardis_stack_desc_t* desc, const void* x, void* y, void* work, void* keep, int64_t n,
                                     cudaStream_t s);   // stack.cu; arguments checked by the caller
tardis_status_t launch_build_predictor(int h, int d, int dtype, const void* W1, const double* U, int bits, int G, uint32_t* codes,
                                       void* scale, uint8_t* zero, cudaStream_t s);   // gptq.cu; arguments checked by the caller
tardis_status_t launch_fold_tensor(Handle* H, const tardis_fold_desc_t* desc, cudaStream_t s);  // bf16 fold on the tensor cores

// ---- small device helpers ----
template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// offline statistics (calibrate.cu)
tardis_status_t launch_neuron_thresholds(int h, int n, const float* z, long long ldz, const float* b1, const float* lo, const float* hi,
                                         int act, double t_layer, double t_min, double t_max, float* err, float* t, cudaStream_t s);
tardis_status_t launch_calibrate(int h, int n, const float* z, long long ldz, const float* b1, double q_lo, double q_hi, int act,
                                 float* lo, float* hi, float* a, float* c, cudaStream_t s);

tardis_status_t launch_range_search(int h, int n, const float* z, long long ldz, const float* b1, const float* thr, double t_all,
                                    double step, int act, float* lo, float* hi, float* a, float* c, int* steps_out, cudaStream_t s);

// the activation (the name is historical: ReLU is served too)
__device__ __forceinline__ float gelu_f32(float z, int act) {
  if (act == TARDIS_ACT_RELU) return z > 0.f ? z : 0.f * z;      // 0 * z keeps NaN a NaN
  if (act == TARDIS_ACT_GELU_TANH) {
    float u = 0.7978845608028654f * (z + 0.044715f * z * z * z);
    return 0.5f * z * (1.0f + tanhf(u));
  }
  return 0.5f * z * (1.0f + erff(z * 0.7071067811865476f));
}
// The tanh form without branches: (1 + tanh u) / 2 = 1 / (1 + e^-2u), with the exponential of -|2u|, so that what is rounded is small beside z.
// (Against 64 bits, root mean square over [-1, 5]: 7.1e-8, of the form with tanhf 9.3e-8; over [-6, -1] 6e-9 against 2.9e-8.)
__device__ __forceinline__ float gelu_tanh_f32(float z) {
  const float e = __expf(-fabsf(z * fmaf(0.0713548162726f, z * z, 1.59576912161f))), half = 0.5f * z;
  return (half + fabsf(half)) - __fdividef(fminf(fabsf(z), 3.0e38f) * e, 1.f + e);       // (halves first: twice z may be too large)
}
__device__ __forceinline__ double gelu_f64(double z, int act) {
  if (act == TARDIS_ACT_RELU) return z > 0.0 ? z : 0.0 * z;
  if (act == TARDIS_ACT_GELU_TANH) {
    // (1 + tanh u) / 2 = 1 / (1 + e^-2u): one exponential and one division, and no cancellation where tanh u is near -1
    const double u2 = 1.5957691216057308 * (z + 0.044715 * z * z * z);
    return z / (1.0 + exp(-u2));
  }
  return 0.5 * z * (1.0 + erf(z * 0.7071067811865476));
}

}  // namespace tardis
