// Shared host/device helpers of the adapshot CUDA library (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "adapshot.h"
#include "rope_theta.h"

#define ADAPSHOT_VERSION_NUMBER 100

#define ADS_CHECK_CUDA(expr)                              \
  do {                                                    \
    cudaError_t e__ = (expr);                             \
    if (e__ != cudaSuccess) return ADAPSHOT_ECUDA;        \
  } while (0)

static inline bool ads_aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline size_t ads_round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// A launch failure is reported as ADAPSHOT_ECUDA without clearing anything else.
static inline int ads_launch_status() {
  return cudaGetLastError() == cudaSuccess ? ADAPSHOT_OK : ADAPSHOT_ECUDA;
}

// Per-device host-side caches: a process may drive several GPUs, and both the SM count and a
// kernel's shared-memory attribute belong to the device that is current at the call.
constexpr int kAdsMaxDevices = 64;
static inline int ads_current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kAdsMaxDevices) return -1;
  return dev;
}
// SM count of the current device (0 on error); looked up once per device.
static inline int ads_sm_count() {
  static int n_sm[kAdsMaxDevices] = {0};
  const int dev = ads_current_device();
  if (dev < 0) return 0;
  if (n_sm[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 0;
    n_sm[dev] = n;
  }
  return n_sm[dev];
}
// Raises a kernel's dynamic shared-memory limit once per device.  `done` is a per-kernel table
// (kAdsMaxDevices entries) owned by the caller.  The value is the same every time, so two
// threads that race here both write it.
template <typename Kernel>
static inline int ads_set_max_smem(Kernel kernel, int bytes, bool* done) {
  const int dev = ads_current_device();
  if (dev < 0) return ADAPSHOT_ECUDA;
  if (!done[dev]) {
    ADS_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    done[dev] = true;
  }
  return ADAPSHOT_OK;
}

// Programmatic dependent launch: the kernel may be started while the one in front of it in the stream still
// ends, so that its launch and its set-up cost no gap (a pass of a few short shots, nine kernels: 45.9 -> 28.3 us; two rounds
// of probes 637 -> 622; a ranking by attention over 2048 shots 912 -> 906).  Every kernel launched this way calls
// ads_dependency_wait(), in every block (what completes a kernel is the completion of its blocks, and a block that did not wait
// would not stand for the kernels before), and before the wait it writes no memory and relies on none.  Only the two decode
// kernels read any there, as a guess: past the L1, so that no old line is left in it for the reads behind the wait; clamped or
// checked so that no address leaves its buffer whatever they find, tiles by L2 prefetches alone; and compared behind the wait with
// what is read there before a result depends on it.  ads_dependency_trigger() lets the next
// kernel in earlier, once all blocks have called it; only the decode kernels do: elsewhere the early blocks took room from
// the kernel they waited for (one layer of one query 132 -> 139 us with triggers in every kernel, the selection's alone
// account for all of it).
template <typename... KArgs, typename... Args>
static inline void ads_launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                        const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);     // (a failure is found by ads_launch_status)
}
__device__ __forceinline__ void ads_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void ads_dependency_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Device: record an error code once; later codes do not overwrite the first.
__device__ __forceinline__ void ads_set_status(int32_t* status, int32_t code) {
  if (status != nullptr) atomicCAS(status, 0, code);
}

// Order-preserving map of an fp64 score to an unsigned key; larger score -> SMALLER key so that an
// ascending order on (key, id) lists the most relevant shot first and equal scores by ascending id.
__device__ __forceinline__ unsigned long long ads_desc_key(double s) {
  unsigned long long u = (unsigned long long)__double_as_longlong(s);
  u = (u >> 63) ? ~u : (u | 0x8000000000000000ull);   // ascending in s
  return ~u;
}
__device__ __forceinline__ double ads_key_score(unsigned long long k) {
  unsigned long long u = ~k;
  u = (u >> 63) ? (u & 0x7fffffffffffffffull) : ~u;
  return __longlong_as_double((long long)u);
}

// Top k of N candidates per query from their sort keys (select.cu): keys [B][N] as ads_desc_key
// writes them; equal keys by the lower index.  Enqueues on st; returns an ADAPSHOT_* code.
int ads_topk_from_keys(const unsigned long long* keys, int N, int B, int k, int32_t* sel_idx, float* sel_score,
                       cudaStream_t st);

// One entropy call, checked and cut into blocks (entropy.cu): what a kernel needs that runs it beside its own work.
struct AdsEntropyJob {
  const void* logits;
  float* partial;              // [blocks][3]
  float* H;
  int32_t* first_ok;
  long long row_stride;
  int f32, R, V, slice, n_split, rows_per_group;
  float tau;
  int blocks;                  // R * n_split; 0: no job
};
int ads_entropy_job(const void* logits, int32_t dtype, int32_t R, int32_t V, int64_t row_stride, float* H, float tau,
                    int32_t rows_per_group, int32_t* first_ok, void* ws, size_t ws_bytes, AdsEntropyJob* job);

// What the calls of a pass share (null, or a null member: nothing).
struct AdsPass {
  const double* theta;         // the model's rotary frequencies
  const AdsEntropyJob* ent;    // the entropy of the probes' logits, to run beside the attention call
};

// The gather (assemble.cu) and the three attention calls (attn.cu) behind their entry points.
int ads_assemble_kv(const adapshot_model_t* model, const adapshot_pool_t* pool, const int32_t* sel_idx, int32_t B, int32_t k,
                    int32_t shot_begin, int32_t layer_begin, int32_t layer_end, void* k_ctx, void* v_ctx, int64_t ctx_cap,
                    int64_t* ctx_off, uint32_t flags, int32_t* status, void* stream, const AdsPass* pass);
int ads_query_attn(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx, int64_t ctx_cap,
                   const int64_t* ctx_off, int32_t B, int32_t k, const int32_t* probe_nshots, int32_t P, const void* q,
                   const void* kq, const void* vq, int32_t Tq, int32_t layer_begin, int32_t layer_end, void* out, float* lse,
                   uint32_t flags, void* ws, size_t ws_bytes, int32_t* status, void* stream, const AdsPass* pass);
int ads_query_attn_fused(const adapshot_model_t* model, const adapshot_pool_t* pool, const int32_t* sel_idx,
                         const int64_t* ctx_off, int64_t ctx_cap, int32_t B, int32_t k, const int32_t* probe_nshots,
                         int32_t P, const void* q, const void* kq, const void* vq, int32_t Tq, int32_t layer_begin,
                         int32_t layer_end, void* out, float* lse, uint32_t flags, void* ws, size_t ws_bytes,
                         int32_t* status, void* stream, const AdsPass* pass);
int ads_query_attn_vpool(const adapshot_model_t* model, const adapshot_pool_t* pool, const int32_t* sel_idx,
                         const void* k_ctx, int64_t ctx_cap, const int64_t* ctx_off, int32_t B, int32_t k,
                         const int32_t* probe_nshots, int32_t P, const void* q, const void* kq, const void* vq, int32_t Tq,
                         int32_t layer_begin, int32_t layer_end, void* out, float* lse, uint32_t flags, void* ws,
                         size_t ws_bytes, int32_t* status, void* stream, const AdsPass* pass);

// Decoding with few rows per KV head (decode.cu): whether a call's rows fit, whether it pays, its scratch, and the call itself
// (arguments checked by the caller).
bool ads_decode_rows_fit(const adapshot_model_t* model, int T_new);
bool ads_decode_rows_pay(const adapshot_model_t* model, int B, int T_new, int T_own, int64_t ctx_cap);
size_t ads_decode_rows_workspace(const adapshot_model_t* model, int B);
int ads_decode_rows(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx, int64_t ctx_cap,
                    const int64_t* ctx_off, int B, int k, const int32_t* n_shots, const void* q_new, const void* k_own,
                    const void* v_own, int T_new, int T_own, int nl, void* out, float* lse, void* ws, int32_t* status,
                    cudaStream_t st);

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Angle p * theta_i formed in fp64 and reduced to [-pi, pi] before the fp32
// sincos, so that the result keeps fp32 accuracy at positions of 64K and more.
__device__ __forceinline__ float rope_reduced_angle(double delta, double theta) {
  const double kInv2Pi = 0.15915494309189533577;
  const double k2PiHi = 6.283185307179586232;
  const double k2PiLo = 2.449293598294706354e-16;
  double a = delta * theta;
  double n = rint(a * kInv2Pi);
  double r = fma(-n, k2PiHi, a);
  r = fma(-n, k2PiLo, r);
  return static_cast<float>(r);
}
__device__ __forceinline__ void rope_sincos(double delta, double theta, float* s, float* c) {
  sincosf(rope_reduced_angle(delta, theta), s, c);
}
// Hardware approximations (absolute error below 1e-6 on [-pi, pi]): for bf16 storage only.
__device__ __forceinline__ void rope_sincos_fast(double delta, double theta, float* s, float* c) {
  const float r = rope_reduced_angle(delta, theta);
  *s = __sinf(r);
  *c = __cosf(r);
}
