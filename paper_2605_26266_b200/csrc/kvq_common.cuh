// Shared host/device helpers of libkvq (internal; not part of the C ABI).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "kvq.h"

namespace kvq {

// Records a failing CUDA runtime call for kvq_last_cuda_error() and maps it to KVQ_ERR_CUDA.
int record_cuda_error(cudaError_t e);

#define KVQ_CUDA_TRY(expr)                                   \
  do {                                                       \
    cudaError_t kvq_e_ = (expr);                             \
    if (kvq_e_ != cudaSuccess) return ::kvq::record_cuda_error(kvq_e_); \
  } while (0)

// Per-device host state.  One process may drive several GPUs, and several threads may call into the library:
// whatever is looked up or configured once is kept per device ordinal, in atomics (a race only repeats an
// idempotent CUDA call).
constexpr int kMaxDevices = 64;
// Ordinal of the calling thread's current device; KVQ_ERR_UNSUPPORTED beyond kMaxDevices.
int current_device(int* dev);
// Multiprocessor count of the current device (looked up once per device).
int device_sm_count(int* sms);
// "Has this been set up on the current device?" for one kernel instantiation: declare one static PerDevice per
// instantiation; first() is true until done() has been called on that device.
struct PerDevice {
  std::atomic<unsigned char> flag[kMaxDevices] = {};
  bool first(int dev) const { return flag[dev].load(std::memory_order_acquire) == 0; }
  void done(int dev) { flag[dev].store(1, std::memory_order_release); }
};

// Shape part of the descriptor check (no pointers).
int check_shape(const kvq_cache_desc* d);
// Shape + the six buffer pointers.
int check_desc(const kvq_cache_desc* d);
int check_tensor(const void* p, kvq_strides s);

inline int groups_of(const kvq_cache_desc* d) { return d->head_dim / d->group; }
inline int code_bytes_of(const kvq_cache_desc* d) { return d->head_dim * d->bits / 8; }

// launchers implemented in the kernel translation units
int launch_quantize_append(const kvq_cache_desc* d, int64_t cache_len, const void* k, const void* v,
                           kvq_strides kv, int64_t n_tokens, cudaStream_t st);
int launch_unpack_codes(const kvq_cache_desc* d, int which, int64_t begin, int64_t n, uint8_t* out,
                        cudaStream_t st);

struct AttnArgs {
  const kvq_cache_desc* desc;
  int64_t cache_begin, cache_len;
  const void* q; kvq_strides qs;
  const void* k_cur; const void* v_cur; kvq_strides kvs;   // strides of k_cur
  kvq_strides vs;                                            // strides of v_cur
  int64_t m_tokens, n_cur;
  void* out; kvq_strides os;
  float softmax_scale;
  uint32_t flags;
  float* lse; float* cached_mass;
  void* workspace; size_t workspace_bytes;
  int32_t* status_word;
  cudaStream_t stream;
};
int launch_attn_mma_sync(const AttnArgs& a);
// Kernel for a few query rows (attn_short.cu), chosen by KVQ_KERNEL_AUTO only.
bool attn_short_supports(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur, uint32_t flags);
size_t attn_short_workspace_bytes(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur);
int attn_short_kernel_launches(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur);
int launch_attn_short(const AttnArgs& a);
// Per-row Jensen-Shannon divergence of the attention weights against those of the BF16 keys k_ref (analysis kernel).
int launch_attn_jsd(const AttnArgs& a, const void* k_ref, kvq_strides ref_strides, float* jsd_out);
// y = (1/sqrt d) H (signs . x) per row (inverse: x = signs . ((1/sqrt d) H y)), BF16 [batch, heads, tokens, head_dim]
int launch_rotate_rows(const kvq_cache_desc* d, const void* src, kvq_strides ss, void* dst, kvq_strides ds,
                       int64_t tokens, bool inverse, cudaStream_t st);
// tcgen05 kernel: returns KVQ_ERR_UNSUPPORTED for shapes it does not cover.
bool attn_tcgen05_supports(const kvq_cache_desc* d, int64_t m_tokens, int64_t n_cur);
// Do the problem's tile steps (one-CTA kernel) fit the kernel's 32-bit counts?
bool attn_tcgen05_counts(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur);
// Can TMA address the call's Q, K_cur, V_cur (no zero stride in a real dimension, byte strides below 2^40)?
bool attn_tcgen05_addressable(const AttnArgs& a);
// pair: the CTA-pair form of the kernel (KVQ_KERNEL_TCGEN05_PAIR), which plans 512-row units over SM pairs
// least: what it can do with, the plan without FP32 partial rows of 128 channels
size_t attn_tcgen05_workspace_bytes(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur, bool pair, bool least = false);
int attn_tcgen05_kernel_launches(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur, bool pair);
int launch_attn_tcgen05(const AttnArgs& a);
// Cycle budget of the tcgen05 kernel's device-side waits for later launches (0 = the default of about a second).
void set_attn_wait_budget(uint32_t cycles);
// Same kernel, partial results of split units in the library's built-in scratch buffer (no caller workspace).
int launch_attn_tcgen05_static(const AttnArgs& a);

#ifdef __CUDACC__
// Launches `kern` so that its blocks may start before the previous kernel in the stream has finished (it waits by itself,
// see wait_for_previous_grid), in clusters of `cluster` blocks; overlap = false: an ordinary launch.
template <typename... Params, typename... Args>
int launch_after(bool overlap, int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st, void (*kern)(Params...), const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (overlap) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr; cfg.numAttrs = n;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  if (e != cudaSuccess) {
    cudaGetLastError();                                // or the next call's ordinary launch would report it again
    return record_cuda_error(e);
  }
  return KVQ_OK;
}

// Kernels overlap (launch_after): one allows the next grid's blocks to start when its own have all started (allow_next_grid), and
// the next waits before it touches what the one before writes.  Every block of a kernel waits, so that work ordered behind it
// is ordered behind the ones before too.  The first kernel of a call is launched this way as well: its blocks are placed, and the
// attention kernel's prologue runs, while the last kernel in the stream, whoever's it is, drains.  It waits before it touches any global
// memory, and only then allows the next grid, so that the call's later kernels may read the caller's tensors without waiting again.
// The wait is for the grid directly before; that one's end implies the end of what lies before it, as with an ordinary launch, unless it
// overlaps that and never waited, which kvq.h therefore asks callers not to put right in front of a call.
// Among other calls on the same inputs (24 heads x 4680 tokens, 16 heads x 1560 rows, 64 heads x 2048 rows, us): append 21.6 ->
// 19.6, attention 125.4 -> 123.6, 64 channels 134.5 -> 130.5, empty cache 167 -> 163.5.
__device__ __forceinline__ void allow_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// How a kernel that waits there reads what a grid before may have written: with an ordinary load.  The read-only path (`__ldg`,
// ld.global.nc) is defined only for memory that nothing writes during the kernel, and such a kernel has started by then; nor does the
// wait hold back loads that the compiler takes for invariant.
template <typename T>
__device__ __forceinline__ T load_coherent(const T* p) {
  __builtin_assume(__isGlobal(p));
  return *p;
}

// ---- device-side number-format helpers -------------------------------------------------

// FP32 -> E4M3 byte, round-to-nearest-even, saturating to +-448 (hardware conversion).
__device__ __forceinline__ uint32_t f32_to_e4m3_byte(float x) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.0f), "f"(x));
  return r & 0xFFu;
}

// E4M3 byte -> FP32 (exact).
__device__ __forceinline__ float e4m3_byte_to_f32(uint32_t b) {
  uint32_t h2;
  uint16_t in = (uint16_t)(b & 0xFFu);
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(in));
  __half lo = __ushort_as_half((unsigned short)(h2 & 0xFFFFu));
  return __half2float(lo);
}

__device__ __forceinline__ float bf16_bits_to_f32(uint32_t bits16) { return __uint_as_float(bits16 << 16); }

__device__ __forceinline__ uint32_t f32_to_bf16_bits(float x) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
}

// A running maximum as the subtrahend of the scores: 0 while all of them were -inf, whose weights are then 0 and not NaN.
__device__ __forceinline__ float no_key_yet(float m) { return m == __int_as_float(0xFF800000) ? 0.f : m; }

// The 16-bit forms of x^ = (code - zero) * step round once, as the FP32 form followed by one conversion does, while their
// constants are exact.  Keys (FP16) and 2-bit values (BF16) subtract (OFF + zero) * step, OFF = 4 or 16, with an FMA: an
// integer of 7 (4) bits times a step of 4 is exact in 11 (8), and with |OFF + zero| up to 112 no key reaches the largest
// FP16 value, where the FP32 form saturates.  4-bit values subtract 16 + zero before the multiplication: exact while code -
// zero and 16 + zero have 8 bits.  False for NaN and infinities.
template <int BITS>
__device__ __forceinline__ bool key_constant_exact(float zero) { return fabsf((BITS == 2 ? 4.f : 16.f) + zero) <= 112.f; }
template <int BITS>
__device__ __forceinline__ bool value_constant_exact(float zero) {
  return BITS == 2 ? fabsf(4.f + zero) <= 16.f : fabsf(16.f + zero - 15.5f) <= 240.5f;
}
#endif

}  // namespace kvq
