// Softmax entropy of last-token logits (paper Eq. 2, over the whole vocabulary)
// and the threshold rule stated after it.
//
// One pass: every thread keeps (m, s, t) with s = sum e^{x-m}, t = sum e^{x-m}(x-m)
// for a running maximum m; states merge exactly (up to rounding) under a change of
// maximum, and H = ln s - t / s at the end.  Rows are split over several CTAs so a
// handful of 128K-entry rows still fills the machine; the per-split states go
// through the caller's workspace and a second, tiny kernel merges them.
#include <float.h>

#include "common.cuh"
#include "entropy.cuh"

namespace {

template <typename T>
__global__ void __launch_bounds__(kEntThreads, 5)
entropy_partial_kernel(const T* __restrict__ logits, int V, long long row_stride, int slice, int n_split,
                       float* __restrict__ partial) {
  ads_dependency_wait();
  // one-dimensional grid: the row count is not bound by the 65535 limit of the other grid dimensions
  ent_partial_block(logits, V, row_stride, slice, n_split, partial, blockIdx.x);
}

__global__ void __launch_bounds__(256)
entropy_finish_kernel(const float* __restrict__ partial, int n_split, int R, int rows_per_group,
                      float tau, float* __restrict__ H, int32_t* __restrict__ first_ok) {
  ads_dependency_wait();
  extern __shared__ float sh_h[];
  ent_finish_block(partial, n_split, R, rows_per_group, tau, H, first_ok, blockIdx.x, sh_h);
}

// Two-token form of Eq. 2 (the paper takes the entropy over the answer tokens {Yes, No}): like
// entropy_finish_kernel, but the sum runs over the `n_subset` listed token ids only.
//   renorm == 0: p_v from the softmax over the whole vocabulary, H = -sum_{v in S} p_v ln p_v
//   renorm == 1: q_v = p_v / sum_{S} p, H = -sum q_v ln q_v
template <typename T>
__global__ void __launch_bounds__(256)
entropy_subset_finish_kernel(const float* __restrict__ partial, int n_split, int R, int rows_per_group,
                             const T* __restrict__ logits, long long row_stride, int V,
                             const int32_t* __restrict__ subset_ids, int n_subset, int renorm,
                             float tau, float* __restrict__ H, int32_t* __restrict__ first_ok,
                             int32_t* __restrict__ status) {
  ads_dependency_wait();
  extern __shared__ float sh_h[];
  const int g = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  for (int j = warp; j < rows_per_group; j += n_warps) {
    const int r = g * rows_per_group + j;
    if (r >= R) break;
    EntState st{-FLT_MAX, 0.f, 0.f};
    for (int s = lane; s < n_split; s += 32) {
      const float* p = partial + 3ll * ((long long)r * n_split + s);
      st = ent_merge(st, EntState{p[0], p[1], p[2]});
    }
    st = ent_warp_reduce(st);
    const float m = __shfl_sync(0xffffffffu, st.m, 0);
    const float ln_s = logf(__shfl_sync(0xffffffffu, st.s, 0));
    const T* row = logits + (long long)r * row_stride;
    float z = 0.f, u = 0.f, h = 0.f;           // sum e^{x-m}, sum e^{x-m}(x-m), -sum p ln p
    for (int i = lane; i < n_subset; i += 32) {
      const int id = subset_ids[i];
      if (id < 0 || id >= V) {
        ads_set_status(status, ADAPSHOT_EINDEX);
        continue;
      }
      float x;
      if constexpr (sizeof(T) == 4) x = row[id]; else x = __bfloat162float(row[id]);
      const float d = x - m;
      const float e = __expf(d);
      z += e;
      u += e > 0.f ? e * d : 0.f;
      const float lp = d - ln_s;                // ln p_v
      const float pv = __expf(lp);
      h -= pv > 0.f ? pv * lp : 0.f;
    }
    z = warp_sum(z); u = warp_sum(u); h = warp_sum(h);
    if (lane == 0) {
      float out = renorm ? (z > 0.f ? logf(z) - u / z : 0.f) : h;
      out = fmaxf(out, 0.f);
      H[r] = out;
      sh_h[j] = out;
    }
  }
  __syncthreads();
  if (first_ok != nullptr && threadIdx.x == 0) {
    int ok = -1;
    for (int j = 0; j < rows_per_group && g * rows_per_group + j < R; ++j) {
      if (sh_h[j] <= tau) { ok = j; break; }
    }
    first_ok[g] = ok;
  }
}

// A fixed figure rather than the SM count of the current device, so that the workspace size
// can be asked for without a device and does not change from one GPU to another: one resident
// wave of 256-thread CTAs at 48 registers (five per SM) on 148 SMs.  (Six per SM at 40 registers, with
// sums added across each vector: 51.9 us for 1024 rows of 128 256 bf16 logits, 188 us for 4096; now 48.7
// and 171 us = 6.1 TB/s.)
constexpr int kEntTargetCtas = 740;
constexpr int kEntSliceUnit = 8192;      // entries: what a CTA's unrolled loop takes per trip (bf16)
constexpr int kEntCtaOverhead = 2048;    // fixed cost of a CTA (start, state merge, store) in entries

// Rows are cut into slices of j * kEntSliceUnit entries (the last one shorter).  A call's CTAs run
// in ceil(R * n / kEntTargetCtas) waves of about equal length (slice + overhead), so the j that
// minimises waves * (slice + overhead) is taken: 1024 rows of 128 256 run as 2 slices each (2.8
// waves) rather than whole (1.4 waves, the second one two fifths full), 224 rows as 3 slices (one wave).  `max_states` bounds R * n (the fixed scratch of the static entry point).
struct EntSplit { int slice, n; };
constexpr int kEntMaxSlices = 64;        // of a row
EntSplit ent_split(int R, int V, long long max_states = 0x7fffffffll) {
  const long long unit = kEntSliceUnit;
  const long long kMaxSlice = 0x7fffe000ll;                             // the largest multiple of the unit an int holds
  EntSplit best{(int)((long long)V <= kMaxSlice ? ((long long)V + unit - 1) / unit * unit : kMaxSlice),
                (long long)V <= kMaxSlice ? 1 : 2};                      // the row in one piece (two beyond 2^31 - 8192)
  double best_cost = 0.0;
  for (int want = 1; want <= kEntMaxSlices; ++want) {
    // the shortest slice (a multiple of the unit) that cuts the row into at most `want` pieces
    const long long per = ((long long)V + want - 1) / want;
    long long slice = (per + unit - 1) / unit * unit;
    if (slice > kMaxSlice) slice = kMaxSlice;
    const int n = (int)(((long long)V + slice - 1) / slice);
    if ((long long)R * n > max_states) break;                            // n only grows with `want`
    const long long waves = ((long long)R * n + kEntTargetCtas - 1) / kEntTargetCtas;
    const double cost = (double)waves * (double)(slice + kEntCtaOverhead);
    if (want == 1 || cost < best_cost) {
      best = EntSplit{(int)slice, n};
      best_cost = cost;
    }
  }
  return best;
}
int ent_splits(int R, int V) { return ent_split(R, V).n; }
size_t ent_state_bytes(long long states) { return ads_round_up((size_t)states * 3 * sizeof(float), 256); }

}  // namespace

extern "C" size_t adapshot_entropy_workspace_bytes(int32_t R, int32_t V) {
  if (R <= 0 || V <= 0) return 0;
  // As many slices as a row of this length is ever cut into: fewer rows are cut into more slices, and a workspace for a
  // batch has to serve every smaller one.
  const long long n = ((long long)V + kEntSliceUnit - 1) / kEntSliceUnit;
  return ent_state_bytes((long long)R * (n < kEntMaxSlices ? n : kEntMaxSlices));
}

int ads_entropy_job(const void* logits, int32_t dtype, int32_t R, int32_t V, int64_t row_stride, float* H, float tau,
                    int32_t rows_per_group, int32_t* first_ok, void* ws, size_t ws_bytes, AdsEntropyJob* job) {
  if (logits == nullptr || H == nullptr || ws == nullptr) return ADAPSHOT_EINVAL;
  if (R <= 0 || V <= 0 || row_stride < V) return ADAPSHOT_EINVAL;
  if (dtype != ADAPSHOT_F32 && dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (rows_per_group <= 0) rows_per_group = 1;
  if (R % rows_per_group != 0 || rows_per_group > 8192) return ADAPSHOT_ESHAPE;
  const EntSplit cut = ent_split(R, V);
  if ((long long)R * cut.n > 0x7fffffffll) return ADAPSHOT_ESHAPE;
  const size_t es = dtype == ADAPSHOT_F32 ? 4 : 2;
  if (!ads_aligned16(logits) || !ads_aligned16(ws) || (row_stride * es) % 16 != 0) return ADAPSHOT_EALIGN;
  if (ws_bytes < ent_state_bytes((long long)R * cut.n)) return ADAPSHOT_ECAPACITY;
  *job = AdsEntropyJob{logits, static_cast<float*>(ws), H, first_ok, row_stride, dtype == ADAPSHOT_F32, R, V, cut.slice, cut.n,
                       rows_per_group, tau, R * cut.n};
  return ADAPSHOT_OK;
}

extern "C" int adapshot_entropy(const void* logits, int32_t dtype, int32_t R, int32_t V,
                                int64_t row_stride, float* H, float tau, int32_t rows_per_group,
                                int32_t* first_ok, void* ws, size_t ws_bytes, int32_t* status,
                                void* stream) {
  (void)status;
  AdsEntropyJob e;
  const int rc = ads_entropy_job(logits, dtype, R, V, row_stride, H, tau, rows_per_group, first_ok, ws, ws_bytes, &e);
  if (rc != ADAPSHOT_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (e.f32)
    ads_launch_dependent(entropy_partial_kernel<float>, (unsigned)e.blocks, kEntThreads, 0, st,
        static_cast<const float*>(logits), V, row_stride, e.slice, e.n_split, e.partial);
  else
    ads_launch_dependent(entropy_partial_kernel<__nv_bfloat16>, (unsigned)e.blocks, kEntThreads, 0, st,
        static_cast<const __nv_bfloat16*>(logits), V, row_stride, e.slice, e.n_split, e.partial);
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  ads_launch_dependent(entropy_finish_kernel, R / e.rows_per_group, 256, e.rows_per_group * sizeof(float), st,
      e.partial, e.n_split, R, e.rows_per_group, tau, H, first_ok);
  return ads_launch_status();
}


extern "C" int adapshot_entropy_subset(const void* logits, int32_t dtype, int32_t R, int32_t V,
                                       int64_t row_stride, const int32_t* subset_ids, int32_t n_subset,
                                       uint32_t flags, float* H, float tau, int32_t rows_per_group,
                                       int32_t* first_ok, void* ws, size_t ws_bytes, int32_t* status,
                                       void* stream) {
  if (logits == nullptr || H == nullptr || ws == nullptr || subset_ids == nullptr) return ADAPSHOT_EINVAL;
  if (R <= 0 || V <= 0 || row_stride < V || n_subset <= 0 || n_subset > V || (flags & ~1u) != 0)
    return ADAPSHOT_EINVAL;
  if (dtype != ADAPSHOT_F32 && dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (rows_per_group <= 0) rows_per_group = 1;
  if (R % rows_per_group != 0 || rows_per_group > 8192) return ADAPSHOT_ESHAPE;
  if ((long long)R * ent_splits(R, V) > 0x7fffffffll) return ADAPSHOT_ESHAPE;
  const size_t es = dtype == ADAPSHOT_F32 ? 4 : 2;
  if (!ads_aligned16(logits) || !ads_aligned16(ws) || (row_stride * es) % 16 != 0 ||
      ((uintptr_t)subset_ids & 3u))
    return ADAPSHOT_EALIGN;
  if (ws_bytes < ent_state_bytes((long long)R * ent_splits(R, V))) return ADAPSHOT_ECAPACITY;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const EntSplit cut = ent_split(R, V);
  const int n_split = cut.n, slice = cut.slice;
  const unsigned grid = (unsigned)((long long)R * n_split);
  float* partial = static_cast<float*>(ws);
  const int renorm = (int)(flags & 1u);
  const size_t sh = rows_per_group * sizeof(float);
  if (dtype == ADAPSHOT_F32) {
    const float* lg = static_cast<const float*>(logits);
    ads_launch_dependent(entropy_partial_kernel<float>, grid, kEntThreads, 0, st, lg, V, row_stride, slice, n_split, partial);
    if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    ads_launch_dependent(entropy_subset_finish_kernel<float>, R / rows_per_group, 256, sh, st,
        partial, n_split, R, rows_per_group, lg, row_stride, V, subset_ids, n_subset, renorm, tau, H, first_ok,
        status);
  } else {
    const __nv_bfloat16* lg = static_cast<const __nv_bfloat16*>(logits);
    ads_launch_dependent(entropy_partial_kernel<__nv_bfloat16>, grid, kEntThreads, 0, st, lg, V, row_stride, slice, n_split, partial);
    if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    ads_launch_dependent(entropy_subset_finish_kernel<__nv_bfloat16>, R / rows_per_group, 256, sh, st,
        partial, n_split, R, rows_per_group, lg, row_stride, V, subset_ids, n_subset, renorm, tau, H, first_ok,
        status);
  }
  return ads_launch_status();
}


// --------------------------------------------------------------------------
// Entropy without any caller-provided or allocated scratch.
//
// Some callers may not allocate device memory at all: code running inside a
// memory-pool-managed serving process whose allocator must not be bypassed, a
// plugin loaded into a host that forbids cudaMalloc after start-up, or a
// latency-critical path where an allocation could synchronise the device.  For
// them the per-split states live in the fixed array below, which every GPU that
// loads this library keeps until the process exits (192 KiB per device).
constexpr int kStaticEntStates = 16384;   // most (row, split) states one call may need
static __device__ __align__(256) float g_entropy_static_scratch[kStaticEntStates * 3];

namespace {
constexpr int kMaxDevices = 64;
float* g_static_scratch_ptr[kMaxDevices] = {nullptr};

// In host code the array's name is only a handle for the runtime; the device
// address has to be asked for, once per device, with that device current.
int static_scratch_for_current_device(float** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ADAPSHOT_ECUDA;
  if (g_static_scratch_ptr[dev] == nullptr) {
    float* ptr = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_entropy_static_scratch) != cudaSuccess ||
        ptr == nullptr)
      return ADAPSHOT_ECUDA;
    g_static_scratch_ptr[dev] = ptr;
  }
  *out = g_static_scratch_ptr[dev];
  return ADAPSHOT_OK;
}
}  // namespace

extern "C" int adapshot_entropy_static(const void* logits, int32_t dtype, int32_t R, int32_t V,
                                       int64_t row_stride, float* H, float tau, int32_t rows_per_group,
                                       int32_t* first_ok, int32_t* status, void* stream) {
  (void)status;
  if (logits == nullptr || H == nullptr) return ADAPSHOT_EINVAL;
  if (R <= 0 || V <= 0 || row_stride < V) return ADAPSHOT_EINVAL;
  if (dtype != ADAPSHOT_F32 && dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (rows_per_group <= 0) rows_per_group = 1;
  if (R % rows_per_group != 0 || rows_per_group > 8192) return ADAPSHOT_ESHAPE;
  if ((long long)R * ent_splits(R, V) > 0x7fffffffll) return ADAPSHOT_ESHAPE;
  const size_t es = dtype == ADAPSHOT_F32 ? 4 : 2;
  if (!ads_aligned16(logits) || (row_stride * es) % 16 != 0) return ADAPSHOT_EALIGN;
  if (R > kStaticEntStates) return ADAPSHOT_ECAPACITY;   // beyond the fixed array
  const EntSplit cut = ent_split(R, V, kStaticEntStates);
  const int n_split = cut.n, slice = cut.slice;

  float* partial = nullptr;
  const int rc = static_scratch_for_current_device(&partial);
  if (rc != ADAPSHOT_OK) return rc;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned grid = (unsigned)((long long)R * n_split);
  // every (row, split) state this call reads is written by the first kernel, so
  // nothing in the shared array has to start at zero
  if (dtype == ADAPSHOT_F32)
    ads_launch_dependent(entropy_partial_kernel<float>, grid, kEntThreads, 0, st,
        static_cast<const float*>(logits), V, row_stride, slice, n_split, partial);
  else
    ads_launch_dependent(entropy_partial_kernel<__nv_bfloat16>, grid, kEntThreads, 0, st,
        static_cast<const __nv_bfloat16*>(logits), V, row_stride, slice, n_split, partial);
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  ads_launch_dependent(entropy_finish_kernel, R / rows_per_group, 256, rows_per_group * sizeof(float), st,
      partial, n_split, R, rows_per_group, tau, H, first_ok);
  return ads_launch_status();
}
