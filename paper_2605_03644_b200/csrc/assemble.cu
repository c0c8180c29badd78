// KV-level concatenation of the selected shots with position re-encoding of K
// (paper Sec. 4.3: Eq. 6 rotary form, Eq. 7 correction by Delta; offsets as in the
// two-shot example, where a shot's Delta is the total length placed before it).
//
// Kernel 1 (plan): ctx_off[b][r] = exclusive prefix sum of the selected lengths.
// Kernel 2 (gather): a selected shot's tokens are consecutive in the pool and in the cache, so both are
// moved by bulk copies, a chunk of consecutive destination tokens at a time: one warp finds the runs of pool
// rows behind a chunk and brings them to shared memory, V leaves from there as it came, K is rotated in place
// by four warps in between.  The rotation angles of a token do not depend on layer or head: a thread forms
// its few (sin, cos) pairs once per chunk, in fp64 before the fp32 sincos, and reuses them.
#include <math.h>

#include <string.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace {

using namespace sm100;

constexpr int kPlanThreads = 256;
constexpr int kTile = 128;   // the attention kernel reads the cache in 128-token tiles
constexpr int kRotWarps = 4;         // gather: warps that rotate K; after them one that loads and one that stores
constexpr int kRotThreads = 32 * kRotWarps;
constexpr int kGatherThreads = kRotThreads + 64;
constexpr int kStages = 3;           // chunks of one CTA on their way at a time
constexpr uint32_t kStageMax = 32768;

// One CTA per query: lengths of the selected shots, block-wide exclusive scan.
__global__ void __launch_bounds__(kPlanThreads)
plan_offsets_kernel(const int32_t* __restrict__ sel_idx, const long long* __restrict__ shot_off,
                    int n_shots, int k, long long ctx_cap, bool check_cap,
                    long long* __restrict__ ctx_off, int32_t* __restrict__ status) {
  __shared__ long long warp_tot[kPlanThreads / 32];
  __shared__ long long carry_sh;
  ads_dependency_wait();
  const int b = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry_sh = 0;
  __syncthreads();
  for (int base = 0; base < k; base += kPlanThreads) {
    const int r = base + threadIdx.x;
    long long len = 0;
    if (r < k) {
      const int s = sel_idx[(long long)b * k + r];
      if (s < 0 || s >= n_shots) ads_set_status(status, ADAPSHOT_EINDEX);
      else len = shot_off[s + 1] - shot_off[s];
    }
    long long incl = len;   // inclusive scan inside the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      long long up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    long long before = carry_sh;
    for (int w = 0; w < warp; ++w) before += warp_tot[w];
    if (r < k) ctx_off[(long long)b * (k + 1) + r] = before + incl - len;
    __syncthreads();
    if (threadIdx.x == kPlanThreads - 1) carry_sh = before + incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const long long L = carry_sh;
    ctx_off[(long long)b * (k + 1) + k] = L;
    if (check_cap && L > ctx_cap) ads_set_status(status, ADAPSHOT_ECAPACITY);
  }
}

template <typename T> struct Vec16;   // one 16-byte vector of T as fp32 lanes
template <> struct Vec16<float> {
  static constexpr int N = 4;
  __device__ static void unpack(const uint4& r, float* x) {
    x[0] = __uint_as_float(r.x); x[1] = __uint_as_float(r.y);
    x[2] = __uint_as_float(r.z); x[3] = __uint_as_float(r.w);
  }
  __device__ static uint4 pack(const float* x) {
    return make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]),
                      __float_as_uint(x[3]));
  }
};
template <> struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void unpack(const uint4& r, float* x) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[2 * j] = __uint_as_float(w[j] << 16);
      x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
  }
  __device__ static uint4 pack(const float* x) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      __nv_bfloat162 h = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);   // round to nearest even
      w[j] = *reinterpret_cast<uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};

struct GatherArgs {
  const void* k_pool;
  const void* v_pool;
  void* k_ctx;
  void* v_ctx;
  const long long* shot_off;
  const int32_t* sel_idx;
  const long long* ctx_off;
  long long pool_tokens;
  long long ctx_cap;
  int n_shots, B, k, n_kv_heads;
  int layer_begin, n_layers_call;
  int shot_begin;              // first selected shot to gather (earlier positions of the cache are kept)
  int k_pos_mode;
  int32_t* status;
  double theta[64];            // theta_i = rope_base^(-2i/D), i < D/2, formed on the host
  int chunk;                   // destination tokens per chunk
  int heads;                   // KV heads per stage (all of them, or rows are cut)
  int layer_groups;            // a chunk's layers are dealt out to this many items
};

// What a stage holds, written by the loading warp.
struct StageInfo {
  long long dst;               // byte offset of the chunk's first row in k_ctx / v_ctx
  long long pos0;              // position of its first token
  int n;                       // tokens; 0: no more stages
  int is_v;
  long long item;              // stages of one item have the same positions
};

// D = head_dim.  A "pair unit" is the 16-byte vector j of the low half of one head
// together with vector j of the high half (elements i and i + D/2 rotate together).
// Bound by HBM.  The copies need no registers and no instructions per byte, so what a CTA has in flight is its
// three stages (two CTAs of 96 KB per SM at the 8B shape; with two stages it is 8-15 % slower), and one layer per
// call moves at the rate of many: the form before, a warp per token with 16-byte loads and stores, had too few
// bytes on their way when the plan lookup and the angles of a token were paid for one or two layers (K only, 32
// queries of 66 K tokens, one layer: 2290 -> 1320 us = 6.5 TB/s; K and V of one layer, 16.4 K tokens: 32 -> 29 us;
// of sixteen layers, 2 K tokens: 55 -> 47 us; K only, four layers, 8 queries of 33 K tokens: 650 -> 663 us).
// WITH_V = false: the K-only form (V is taken from the pool by its consumer).
template <typename T, int D, bool WITH_V>
__global__ void __launch_bounds__(kGatherThreads, 2)
gather_rope_kernel(const __grid_constant__ GatherArgs a) {
  constexpr int EPV = Vec16<T>::N;                 // elements per 16-byte vector
  constexpr int HALF_V = D / EPV / 2;              // pair units per head
  constexpr int kHeadBytes = D * (int)sizeof(T);
  constexpr int kPassTokens = kRotThreads / HALF_V;  // tokens the rotating threads cover at once
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ StageInfo info[kStages];
  __shared__ int first_s[kStages][4 * kPassTokens];  // first position of the shot a token lies in (k_pos_mode 1)
  __shared__ __align__(8) unsigned long long bars[3 * kStages];
  __shared__ int abort_s[2];
  const uint32_t bar0 = smem_u32(bars), smem0 = smem_u32(smem);
  auto full = [&](int s) { return bar0 + 8u * s; };                     // the chunk has landed
  auto done = [&](int s) { return bar0 + 8u * (kStages + s); };         // K has been rotated
  auto empty = [&](int s) { return bar0 + 8u * (2 * kStages + s); };    // the chunk has left
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t stage_bytes = (uint32_t)a.chunk * a.heads * kHeadBytes;
  const int row_bytes = a.n_kv_heads * kHeadBytes;
  const int part_bytes = a.heads * kHeadBytes;     // of a row, in one stage
  const bool cut_rows = a.heads != a.n_kv_heads;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(done(s), kRotWarps);
      mbar_init(empty(s), 1);
    }
    abort_s[0] = abort_s[1] = 0;
    mbar_fence_init();
  }
  __syncthreads();
  ads_dependency_wait();

  if (warp == kRotWarps) {
    // ---------------------------------------------------------------- loading warp
    // A query's chunks that hold a position to gather or to clear, [c0, c0 + n), are all that is dealt out: the capacity
    // behind a query's last token and the prefix that stays (shot_begin) would cost a step of this warp per chunk
    // (half a microsecond each: the last 8 of 512 shots of 32 queries of 66 K tokens, four
    // layers of K: 754 -> 101 us, one layer 200 -> 38).  Lane i knows the i-th of the 32 queries it is at.
    const int group_layers = (a.n_layers_call + a.layer_groups - 1) / a.layer_groups;
    long long q_len = 0, q_begin = 0, q_end = 0, q_c0 = 0;   // tokens, first position, chunks up to this query's end, c0 - chunks before it
    int q0 = 0;
    auto load_queries = [&](int first_query, long long before) {
      q0 = first_query;
      long long n = 0, c0 = 0;
      if (q0 + lane < a.B) {
        const long long* off = a.ctx_off + (long long)(q0 + lane) * (a.k + 1);
        q_len = off[a.k];
        q_begin = off[a.shot_begin];
        c0 = q_begin / a.chunk;
        n = (min((q_len + kTile - 1) / kTile * kTile, a.ctx_cap) + a.chunk - 1) / a.chunk - c0;
        if (n < 0) n = 0;
      }
      q_end = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const long long o = __shfl_up_sync(0xffffffffu, q_end, d);
        if (lane >= d) q_end += o;
      }
      q_end += before;
      q_c0 = c0 - (q_end - n);
    };
    long long total_chunks = 0;
    for (int q = 0; q < a.B; q += 32) {
      load_queries(q, total_chunks);
      total_chunks = __shfl_sync(0xffffffffu, q_end, 31);
    }
    if (a.B > 32) load_queries(0, 0);
    uint32_t it = 0;
    bool ok = true;
    // item = (chunk x, layer group lg), the groups of a chunk side by side: neighbouring CTAs take the same chunk's layers
    long long x = blockIdx.x / a.layer_groups;
    int lg = blockIdx.x % a.layer_groups;
    const int step_x = gridDim.x / a.layer_groups, step_lg = gridDim.x % a.layer_groups;
    for (; x < total_chunks && ok; x += step_x, lg += step_lg) {
      if (lg >= a.layer_groups) {
        lg -= a.layer_groups;
        if (++x >= total_chunks) break;
      }
      for (long long e = __shfl_sync(0xffffffffu, q_end, 31); x >= e; e = __shfl_sync(0xffffffffu, q_end, 31))
        load_queries(q0 + 32, e);
      const int qi = __popc(__ballot_sync(0xffffffffu, q_end <= x));
      const int b = q0 + qi;
      const int l0 = lg * group_layers;
      const int l1 = min(a.n_layers_call, l0 + group_layers);
      const long long p0 = (__shfl_sync(0xffffffffu, q_c0, qi) + x) * a.chunk;
      const long long* off = a.ctx_off + (long long)b * (a.k + 1);
      const long long L = __shfl_sync(0xffffffffu, q_len, qi);
      const long long pa = max(p0, __shfl_sync(0xffffffffu, q_begin, qi));      // positions before it stay as they are
      const long long pb = min(p0 + a.chunk, min(L, a.ctx_cap));
      // zeros for the rest of the last 128-token tile, so that whole tiles can be read later
      const long long za = max(p0, L), zb = min(p0 + a.chunk, min((L + kTile - 1) / kTile * kTile, a.ctx_cap));
      for (int l = l0; za < zb && l < l1; ++l) {
        const long long dst = (((long long)b * a.n_layers_call + l) * a.ctx_cap + za) * row_bytes;
        for (long long v = lane; v < (zb - za) * row_bytes / 16; v += 32) {
          reinterpret_cast<uint4*>(static_cast<char*>(a.k_ctx) + dst)[v] = make_uint4(0, 0, 0, 0);
          if (WITH_V) reinterpret_cast<uint4*>(static_cast<char*>(a.v_ctx) + dst)[v] = make_uint4(0, 0, 0, 0);
        }
      }
      if (pa >= pb) continue;
      // the largest slot in [0, k) with off[slot] <= pa, by a 32-ary search of the whole warp
      int lo = 0, seg_n = a.k;
      while (seg_n > 1) {
        const int stride = (seg_n + 31) / 32;
        const int idx = lo + lane * stride;
        const bool le = idx < lo + seg_n && off[idx] <= pa;
        const int cnt = __popc(__ballot_sync(0xffffffffu, le));        // probes are ascending: a prefix is true
        const int first = lo + (cnt - 1) * stride;                      // cnt >= 1: off[lo] <= pa
        seg_n = min(stride, lo + seg_n - first);
        lo = first;
      }
      // Lane i takes the run of slot lo + i (and of the 32nd after it, ... in chunks of many short shots).
      long long run_src = 0;                       // pool token of the run's first row
      int run_at = 0, run_n = 0, run_first = 0;    // its place in the chunk, its length, its shot's first position
      auto find_run = [&](int group) -> bool {     // whether a further group is needed
        const int slot = lo + 32 * group + lane;
        run_n = 0;
        bool in = slot < a.k;
        const long long o = in ? off[slot] : 0;
        in = in && o < pb;
        if (in) {
          const long long s0 = max(o, pa), s1 = min(off[slot + 1], pb);
          const int s = a.sel_idx[(long long)b * a.k + slot];
          if (s1 > s0 && s >= 0 && s < a.n_shots) {          // (an unknown shot is reported by the plan kernel)
            run_src = a.shot_off[s] + (s0 - o);
            run_at = (int)(s0 - pa);
            run_n = (int)(s1 - s0);
            run_first = (int)o;
          }
        }
        return (__ballot_sync(0xffffffffu, in) >> 31) != 0;
      };
      const bool many = find_run(0);
      int total = __reduce_add_sync(0xffffffffu, run_n);     // tokens that will come
      if (many) {
        bool more = true;
        for (int g = 1; more; ++g) {
          more = find_run(g);
          total += __reduce_add_sync(0xffffffffu, run_n);
        }
        find_run(0);
      }
      for (int l = l0; l < l1 && ok; ++l)
        for (int v = 0; v < (WITH_V ? 2 : 1) && ok; ++v)
          for (int h0 = 0; h0 < a.n_kv_heads; h0 += a.heads, ++it) {
            const int s = it % kStages;
            ok = __all_sync(0xffffffffu, mbar_wait(empty(s), ((it / kStages) & 1) ^ 1, abort_s));
            if (!ok) break;
            const int width = min(a.heads, a.n_kv_heads - h0) * kHeadBytes;
            const char* src = static_cast<const char*>(v ? a.v_pool : a.k_pool) +
                              (long long)(a.layer_begin + l) * a.pool_tokens * row_bytes + h0 * kHeadBytes;
            if (lane == 0) {
              StageInfo& si = info[s];
              si.dst = (((long long)b * a.n_layers_call + l) * a.ctx_cap + pa) * row_bytes + h0 * kHeadBytes;
              si.pos0 = pa;
              si.n = (int)(pb - pa);
              si.is_v = v;
              si.item = x * a.layer_groups + lg;
            }
            if (a.k_pos_mode == 1) {
              bool more = many;
              for (int t = 0; t < run_n; ++t) first_s[s][run_at + t] = run_first;
              for (int g = 1; more; ++g) {
                more = find_run(g);
                for (int t = 0; t < run_n; ++t) first_s[s][run_at + t] = run_first;
              }
              if (many) find_run(0);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive_expect_tx(full(s), (uint32_t)total * width);
            __syncwarp();
            bool more = true;
            for (int g = 0; more; ++g) {
              more = many && (g == 0 || find_run(g));
              const uint32_t dst = smem0 + s * stage_bytes + run_at * part_bytes;
              if (!cut_rows) {
                if (run_n > 0) bulk_load(dst, src + run_src * row_bytes, (uint32_t)run_n * row_bytes, full(s));
              } else {
                for (int t = 0; t < run_n; ++t) bulk_load(dst + t * part_bytes, src + (run_src + t) * row_bytes, width, full(s));
              }
            }
            if (many) find_run(0);
          }
    }
    if (lane == 0) {
      // the end: an empty stage; after giving up, the copies still on their way have to land
      const int s = it % kStages;
      if (ok && mbar_wait(empty(s), ((it / kStages) & 1) ^ 1, abort_s)) {
        info[s].n = 0;
        mbar_arrive(full(s));
      } else {
        for (uint32_t t = it > (uint32_t)kStages ? it - kStages : 0; t < it; ++t)
          mbar_wait(full(t % kStages), (t / kStages) & 1, abort_s + 1);
      }
    }
    __syncwarp();
  } else if (warp == kRotWarps + 1) {
    // ---------------------------------------------------------------- storing warp (one thread)
    if (lane == 0) {
      for (uint32_t it = 0;; ++it) {
        const int s = it % kStages;
        if (!mbar_wait(full(s), (it / kStages) & 1, abort_s)) break;
        const StageInfo si = info[s];
        if (si.n == 0) break;
        // (consumers arrive for every stage, so that the phases of `done` follow those of `full`)
        if (!mbar_wait(done(s), (it / kStages) & 1, abort_s)) break;
        char* dst = static_cast<char*>(si.is_v ? a.v_ctx : a.k_ctx) + si.dst;
        const uint32_t src = smem0 + s * stage_bytes;
        if (!cut_rows) {
          bulk_store(dst, src, (uint32_t)si.n * row_bytes);
        } else {
          const int width = min(part_bytes, row_bytes - (int)(si.dst % row_bytes));
          for (int t = 0; t < si.n; ++t) bulk_store(dst + (long long)t * row_bytes, src + t * part_bytes, width);
        }
        bulk_commit();
        if (it > 0) {                              // the stage before has been read
          bulk_wait_read<1>();
          mbar_arrive(empty((it - 1) % kStages));
        }
      }
      bulk_wait_all();
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- rotating warps
    const int jcol = threadIdx.x % HALF_V, tok0 = threadIdx.x / HALF_V;
    double theta[EPV];
#pragma unroll
    for (int e = 0; e < EPV; ++e) theta[e] = a.theta[jcol * EPV + e];
    float sn[EPV], cs[EPV];
    const bool one_pass = a.chunk <= kPassTokens;
    long long last_item = -1;
    for (uint32_t it = 0;; ++it) {
      const int s = it % kStages;
      if (!__all_sync(0xffffffffu, mbar_wait(full(s), (it / kStages) & 1, abort_s))) break;
      const StageInfo si = info[s];
      if (si.n == 0) break;
      if (!si.is_v) {
        for (int t = tok0; t < si.n; t += kPassTokens) {
          if (!one_pass || si.item != last_item) {
            const double delta = a.k_pos_mode == 0 ? (double)(si.pos0 + t) : (double)first_s[s][t];
#pragma unroll
            for (int e = 0; e < EPV; ++e) {
              // bf16 storage rounds at 2^-9: the hardware sin/cos of the reduced angle is ample there
              if constexpr (sizeof(T) == 2) rope_sincos_fast(delta, theta[e], &sn[e], &cs[e]);
              else rope_sincos(delta, theta[e], &sn[e], &cs[e]);
            }
          }
          unsigned char* row = smem + s * stage_bytes + t * part_bytes + jcol * 16;
#pragma unroll 4
          for (int h = 0; h < a.heads; ++h, row += kHeadBytes) {
            uint4* lo_p = reinterpret_cast<uint4*>(row);
            uint4* hi_p = reinterpret_cast<uint4*>(row + kHeadBytes / 2);
            float x[EPV], y[EPV], xr[EPV], yr[EPV];
            Vec16<T>::unpack(*lo_p, x);
            Vec16<T>::unpack(*hi_p, y);
#pragma unroll
            for (int e = 0; e < EPV; ++e) {
              xr[e] = x[e] * cs[e] - y[e] * sn[e];
              yr[e] = y[e] * cs[e] + x[e] * sn[e];
            }
            *lo_p = Vec16<T>::pack(xr);
            *hi_p = Vec16<T>::pack(yr);
          }
        }
        last_item = si.item;
        fence_proxy_async_smem();                  // the rotated rows, for the bulk store
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(done(s));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && abort_s[0] != 0) ads_set_status(a.status, ADAPSHOT_ETIMEOUT);
}

template <typename T, int D>
int launch_gather(GatherArgs a, cudaStream_t st) {
  constexpr int kPassTokens = kRotThreads / (D / Vec16<T>::N / 2);
  const int n_sm = ads_sm_count();
  if (n_sm <= 0) return ADAPSHOT_ECUDA;
  // A pass of the rotating threads over one head is 4 KB whatever D and T: eight heads fill a stage, more are
  // cut into several stages, fewer leave room for up to four passes (as long as every CTA gets a chunk).
  a.heads = a.n_kv_heads < 8 ? a.n_kv_heads : 8;
  int passes = 8 / a.heads < 4 ? 8 / a.heads : 4;
  auto chunks = [&]() { return (long long)a.B * ((a.ctx_cap + (long long)kPassTokens * passes - 1) / (kPassTokens * passes)); };
  while (passes > 1 && chunks() < 2 * n_sm) passes >>= 1;
  a.chunk = kPassTokens * passes;
  const uint32_t smem = kStages * (uint32_t)a.chunk * a.heads * D * sizeof(T);
  int per_sm = (int)(200 * 1024 / (smem + 4096));
  per_sm = per_sm > 8 ? 8 : per_sm;
  const long long ctas = (long long)n_sm * per_sm;
  // K alone: one item per layer (neighbouring CTAs then take the same chunk's layers; 663 against 687 us for four
  // layers of 8 x 33 K tokens).  With V a chunk's layers stay together (246 against 252 us for three layers of 64 K
  // tokens) unless pairs of them are needed to give every CTA several items.
  long long groups = a.v_ctx == nullptr ? a.n_layers_call : (4 * ctas + chunks() - 1) / chunks();
  if (a.v_ctx != nullptr && groups > (a.n_layers_call + 1) / 2) groups = (a.n_layers_call + 1) / 2;
  a.layer_groups = groups < 1 ? 1 : (int)groups;
  const long long items = chunks() * a.layer_groups;
  const unsigned grid = (unsigned)(items < ctas ? items : ctas);
  static bool attr_done[2][kAdsMaxDevices] = {{false}, {false}};
  const int most = (int)(kStages * kStageMax);
  if (a.v_ctx != nullptr) {
    if (ads_set_max_smem(gather_rope_kernel<T, D, true>, most, attr_done[0]) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    ads_launch_dependent(gather_rope_kernel<T, D, true>, grid, kGatherThreads, smem, st, a);
  } else {
    if (ads_set_max_smem(gather_rope_kernel<T, D, false>, most, attr_done[1]) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    ads_launch_dependent(gather_rope_kernel<T, D, false>, grid, kGatherThreads, smem, st, a);
  }
  return ads_launch_status();
}

}  // namespace

int ads_assemble_kv(const adapshot_model_t* model, const adapshot_pool_t* pool, const int32_t* sel_idx, int32_t B, int32_t k,
                    int32_t shot_begin, int32_t layer_begin, int32_t layer_end, void* k_ctx, void* v_ctx, int64_t ctx_cap,
                    int64_t* ctx_off, uint32_t flags, int32_t* status, void* stream, const AdsPass* pass) {
  if (model == nullptr || pool == nullptr || sel_idx == nullptr || ctx_off == nullptr) return ADAPSHOT_EINVAL;
  if (shot_begin < 0 || shot_begin >= k) return ADAPSHOT_ESHAPE;
  if (B <= 0 || (flags & ~(ADAPSHOT_ASSEMBLE_KEEP_PLAN | ADAPSHOT_ASSEMBLE_K_ONLY)) != 0 ||
      pool->shot_off == nullptr || pool->n_shots <= 0)
    return ADAPSHOT_EINVAL;
  const bool k_only = (flags & ADAPSHOT_ASSEMBLE_K_ONLY) != 0;
  if (k_only) v_ctx = nullptr;
  if (k < 1 || k > pool->n_shots) return ADAPSHOT_ESHAPE;
  const bool plan_only = k_ctx == nullptr && v_ctx == nullptr;
  const bool keep_plan = (flags & ADAPSHOT_ASSEMBLE_KEEP_PLAN) != 0;
  if (plan_only && keep_plan) return ADAPSHOT_EINVAL;
  if (!plan_only && (k_ctx == nullptr || (v_ctx == nullptr && !k_only))) return ADAPSHOT_EINVAL;
  if (((uintptr_t)sel_idx & 3u) || ((uintptr_t)ctx_off & 7u)) return ADAPSHOT_EALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  if (!plan_only) {
    if (pool->k == nullptr || (pool->v == nullptr && !k_only)) return ADAPSHOT_EINVAL;
    if (model->head_dim != 64 && model->head_dim != 128) return ADAPSHOT_ESHAPE;
    if (model->n_kv_heads <= 0 || model->n_q_heads % model->n_kv_heads != 0) return ADAPSHOT_ESHAPE;
    if (layer_begin < 0 || layer_end <= layer_begin || layer_end > model->n_layers) return ADAPSHOT_ESHAPE;
    if (ctx_cap <= 0 || pool->pool_tokens <= 0) return ADAPSHOT_EINVAL;
    if (model->dtype != ADAPSHOT_F32 && model->dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
    if (model->k_pos_mode != 0 && model->k_pos_mode != 1) return ADAPSHOT_EUNSUPPORTED;
    if (!(model->rope_base > 1.0)) return ADAPSHOT_EINVAL;
    if (!ads_aligned16(pool->k) || (!k_only && !ads_aligned16(pool->v)) || !ads_aligned16(k_ctx) ||
        !ads_aligned16(v_ctx))
      return ADAPSHOT_EALIGN;
  }

  if (!keep_plan) {
    ads_launch_dependent(plan_offsets_kernel, B, kPlanThreads, 0, st,
        sel_idx, reinterpret_cast<const long long*>(pool->shot_off), pool->n_shots, k, ctx_cap, ctx_cap > 0,
        reinterpret_cast<long long*>(ctx_off), status);
    if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  }
  if (plan_only) return ADAPSHOT_OK;

  GatherArgs a;
  a.k_pool = pool->k; a.v_pool = pool->v; a.k_ctx = k_ctx; a.v_ctx = v_ctx;
  a.shot_off = reinterpret_cast<const long long*>(pool->shot_off);
  a.sel_idx = sel_idx;
  a.ctx_off = reinterpret_cast<const long long*>(ctx_off);
  a.pool_tokens = pool->pool_tokens; a.ctx_cap = ctx_cap;
  a.n_shots = pool->n_shots; a.B = B; a.k = k; a.n_kv_heads = model->n_kv_heads;
  a.layer_begin = layer_begin; a.n_layers_call = layer_end - layer_begin;
  a.shot_begin = shot_begin;
  a.k_pos_mode = model->k_pos_mode; a.status = status;
  if (pass != nullptr && pass->theta != nullptr) memcpy(a.theta, pass->theta, model->head_dim / 2 * sizeof(double));
  else ads_rope_theta(model->rope_base, model->head_dim, a.theta);

  const bool f32 = model->dtype == ADAPSHOT_F32;
  if (model->head_dim == 128)
    return f32 ? launch_gather<float, 128>(a, st) : launch_gather<__nv_bfloat16, 128>(a, st);
  return f32 ? launch_gather<float, 64>(a, st) : launch_gather<__nv_bfloat16, 64>(a, st);
}

extern "C" int adapshot_assemble_kv(const adapshot_model_t* model, const adapshot_pool_t* pool,
                                    const int32_t* sel_idx, int32_t B, int32_t k,
                                    int32_t layer_begin, int32_t layer_end, void* k_ctx, void* v_ctx,
                                    int64_t ctx_cap, int64_t* ctx_off, uint32_t flags,
                                    int32_t* status, void* stream) {
  return ads_assemble_kv(model, pool, sel_idx, B, k, 0, layer_begin, layer_end, k_ctx, v_ctx, ctx_cap, ctx_off, flags, status,
                         stream, nullptr);
}

extern "C" int adapshot_assemble_kv_from(const adapshot_model_t* model, const adapshot_pool_t* pool,
                                         const int32_t* sel_idx, int32_t B, int32_t k, int32_t shot_begin,
                                         int32_t layer_begin, int32_t layer_end, void* k_ctx, void* v_ctx,
                                         int64_t ctx_cap, int64_t* ctx_off, uint32_t flags,
                                         int32_t* status, void* stream) {
  return ads_assemble_kv(model, pool, sel_idx, B, k, shot_begin, layer_begin, layer_end, k_ctx, v_ctx, ctx_cap, ctx_off, flags,
                         status, stream, nullptr);
}
