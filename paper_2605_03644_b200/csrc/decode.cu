// Decoding over the chosen prefix (paper Sec. 4.1: the shot count that met the threshold is "used for
// subsequent formal inference"): attention of a few new tokens per request over its context and its own
// tokens (Eq. 1, causal among the own tokens), for calls whose rows per KV head (T_new * G) fit 32 (up to 16 always, more
// where it pays).
//
// What bounds it: the K/V bytes (4 * Hkv * d per token; 0.5 to 4 flops per byte and row).  The 128-row tiles of the
// prefill kernel spend a full score tile, softmax and read-out per 128 keys on G rows, and a call is three
// kernels.  Here one kernel streams K and V and does everything else beside them:
//   - the tiles (64 keys of one KV head) of all (request, layer, KV head) units form one sequence that is cut
//     into equal ranges, one per CTA, two CTAs per SM (one CTA's start-up and read-out run under the other's
//     loads; 192 KB of tiles in flight per SM);
//   - one producer thread keeps a ring of TMA tiles full; each of four warps takes 16 of a tile's 64 keys with
//     a running maximum of its own, so that no warp waits for another between two read-outs.  The rows
//     are the 16-row operand of warp-level mma: with so few rows the tensor pipe's rate is not what counts,
//     and the scores stay in registers;
//   - Q is rotated by the CTA that needs it, the own keys in shared memory by the warp that reads them: no
//     preparation kernel and no schedule in memory.
// A unit that a range boundary cuts leaves un-normalised partials, merged by decode_combine_kernel.
// Measured at 32 query / 8 KV heads, d = 128, one layer per call, against the prefill kernels that took these
// calls before: 32 requests of 6 to 16 K tokens (1.6 GB of K/V) 376 -> 256 us = 6.4 TB/s, the copy bandwidth; one request
// (50 MB) 50 -> 14.5 us per call, most of them a chain of latencies that no size makes shorter: launch, the unit's
// look-up, Q, first tiles, merge, and the ends of two kernels.
#include <cuda.h>
#include <math.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.cuh"

namespace {

using namespace sm100;

constexpr int kWarps = 4;                    // consumer warps; warp 4 is the producer
constexpr int kThreads = 32 * (kWarps + 1);
constexpr int kTile = 64;                    // keys per tile, 16 per consumer warp
constexpr int kMaxB = 256;
constexpr int kMaxCtas = 320;                // two per SM, at most this many
constexpr int kUnitCost = 1;                 // fixed cost of a unit (rotate Q, merge the warps), in tiles
constexpr int kMinRange = 3;                 // shortest range, in tiles (fixed cost included)
constexpr int kPrefetchRange = 16;           // ranges of up to this many tiles have their first ones prefetched (32 long requests: 536.7 with, 535.2 without)
constexpr int kPrefetchTiles = 3;            // of a range, brought to L2 ahead (none / 3 / 6 / 12: 67.1 / 63.9 / 64 / 64 us; 32 requests 537 / 537 / 538 / 541)
constexpr int kRows = 32;                    // rows a partial has room for
constexpr int kMergeRows = 4;                // rows whose states the warps merge at a time
constexpr float kNegSentinel = -1.0e30f;
constexpr float kLn2 = 0.6931471805599453f;

template <int D> constexpr int kStages = D == 128 ? 3 : 6;

struct DecodeParams {
  const __nv_bfloat16* q;      // [B][nl][T_new][Hq][D]
  __nv_bfloat16* out;          // like q
  float* lse;                  // [B][nl][Hq][T_new] or null
  float* o_part;               // [2 * n_cta][kRows][D]
  float* ml_part;              // [2 * n_cta][kRows][2]
  long long* prefix;           // [B + 1]: cost of the requests before b, in tiles of one (layer, head) unit
  const long long* ctx_off;    // [B][k + 1]
  const int32_t* n_shots;      // [B]
  int32_t* status;
  long long ctx_cap;
  int B, k, Hq, Hkv, G, nl, T_new, T_own, rows, n_cta;
  float scale_log2;
  double theta[64];
};

// a / b for 0 <= a, 0 < b; the positions of most calls fit 32 bits, where a division is a tenth of the instructions
__device__ __forceinline__ long long div_nn(long long a, long long b) {
  if (((a | b) >> 32) == 0) return (uint32_t)a / (uint32_t)b;
  return a / b;
}

// The part of the tile sequence a CTA takes: every unit (request, layer, KV head) counts its tiles and
// kUnitCost more in front of them.
struct Ranges {
  long long total;
  int n;                       // ranges that are not empty
  __device__ long long start(long long c) const { return c >= n ? total : div_nn(c * total, n); }
  // the range that holds position x (0 <= x < total)
  __device__ int holder(long long x) const { return (int)div_nn((x + 1) * n - 1, total); }
};
__device__ __forceinline__ Ranges make_ranges(long long total, int n_cta) {
  const long long fit = div_nn(total, kMinRange);
  return Ranges{total, (int)(fit < 1 ? 1 : (fit < n_cta ? fit : n_cta))};
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// c (16 x 8, fp32) += a (16 x 16, bf16) b (16 x 8, bf16)
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// barrier of the consumer warps that tells whether every thread's `ok` was set
__device__ __forceinline__ bool consumers_all(bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"(ok ? 1u : 0u) : "memory");
  return r != 0;
}
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

template <int D>
struct DecodeSmem {
  static constexpr uint32_t kTileBytes = kTile * D * 2;          // K or V of one tile
  static constexpr uint32_t kStageBytes = 2 * kTileBytes;
  static constexpr int kQStride = D + 8;                         // elements; rows of Q do not share banks
  static constexpr int kOStride = D + 8;                         // floats; a warp's rows in the merge area
  static constexpr uint32_t kOffQ = kStages<D> * kStageBytes;    // Q of the unit; its read-out merges the warps here
  static constexpr uint32_t kQBytes = kRows * kQStride * 2;
  static_assert(kWarps * kMergeRows * kOStride * 4 <= kQBytes, "the merge area takes the place of Q");
  static constexpr uint32_t kOffRed = kOffQ + kQBytes;           // [kWarps][kMergeRows] row maxima and sums
  static constexpr uint32_t kOffPre = kOffRed + kWarps * kMergeRows * 8;
  static constexpr uint32_t kOffLen = kOffPre + (kMaxB + 1) * 8; // context lengths
  static constexpr uint32_t kOffShots = kOffLen + kMaxB * 4;     // shot counts
  static constexpr uint32_t kOffBar = kOffShots + kMaxB * 4;
  static constexpr uint32_t kTotal = kOffBar + 128 + 1024;       // + alignment slack
};

// MB: blocks of 16 rows (1: T_new * G <= 16, 2: <= 32).
template <int D, int MB>
__global__ void __launch_bounds__(kThreads, 2)
decode_rows_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const __grid_constant__ CUtensorMap tm_ko, const __grid_constant__ CUtensorMap tm_vo,
                   const __grid_constant__ DecodeParams p) {
  using SM = DecodeSmem<D>;
  constexpr int ST = kStages<D>, SUB = D / 64;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_raw + (base - raw_addr);
  __nv_bfloat16* q_s = reinterpret_cast<__nv_bfloat16*>(base_ptr + SM::kOffQ);
  float* o_s = reinterpret_cast<float*>(base_ptr + SM::kOffQ);
  float2* red = reinterpret_cast<float2*>(base_ptr + SM::kOffRed);
  long long* pre = reinterpret_cast<long long*>(base_ptr + SM::kOffPre);
  int* len_s = reinterpret_cast<int*>(base_ptr + SM::kOffLen);
  int* n_s = reinterpret_cast<int*>(base_ptr + SM::kOffShots);
  auto full = [&](int s) { return base + SM::kOffBar + 8u * s; };
  auto empty = [&](int s) { return base + SM::kOffBar + 8u * (ST + s); };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + SM::kOffBar + 16 * ST);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_own = (p.T_own + kTile - 1) / kTile;
  const long long upb = (long long)p.nl * p.Hkv;                 // units per request

  if (threadIdx.x == 128) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), kWarps);
    }
    abort_flag[0] = abort_flag[1] = 0;
    mbar_fence_init();
  }
  ads_dependency_trigger();
  // Context lengths and prefix sums of the requests' costs: every CTA forms them for itself (B <= 256), the loads of
  // all requests on their way at once.  As a guess (before the kernels in front are through) the values are read past the L1
  // and clamped without a report.
  auto clamp_len = [&](long long L) { return L > p.ctx_cap ? p.ctx_cap : (L < 0 ? 0 : L); };
  auto lengths = [&](bool guess) {
    int n[kMaxB / 32];
    long long L[kMaxB / 32];
#pragma unroll
    for (int e = 0; e < kMaxB / 32; ++e)
      if (e * 32 < p.B) n[e] = e * 32 + lane < p.B ? (guess ? __ldcg(p.n_shots + e * 32 + lane) : p.n_shots[e * 32 + lane]) : 1;
#pragma unroll
    for (int e = 0; e < kMaxB / 32; ++e) {
      if (e * 32 >= p.B) break;
      if (n[e] < 1 || n[e] > p.k) {               // reported and clamped
        if (!guess) ads_set_status(p.status, ADAPSHOT_EINDEX);
        n[e] = n[e] < 1 ? 1 : p.k;
      }
      const int b = e * 32 + lane;
      const long long* off = p.ctx_off + (long long)b * (p.k + 1) + n[e];
      L[e] = b < p.B ? (guess ? __ldcg(off) : *off) : 0;
    }
    long long carry = 0;
    if (lane == 0) pre[0] = 0;
#pragma unroll
    for (int e = 0; e < kMaxB / 32; ++e) {
      const int b = e * 32 + lane;
      if (e * 32 >= p.B) break;
      L[e] = clamp_len(L[e]);
      long long v = b < p.B ? (L[e] + kTile - 1) / kTile + n_own + kUnitCost : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      v += carry;
      carry = __shfl_sync(0xffffffffu, v, 31);
      if (b < p.B) {
        len_s[b] = (int)L[e];
        n_s[b] = n[e];
        pre[b + 1] = v;
      }
    }
  };
  // Whether the guess holds: both loads of every request at once, instead of one after the other.
  auto guess_holds = [&]() -> bool {
    int n[kMaxB / 32];
    long long L[kMaxB / 32];
#pragma unroll
    for (int e = 0; e < kMaxB / 32; ++e) {
      const int b = e * 32 + lane;
      if (e * 32 >= p.B) break;
      if (b < p.B) {
        n[e] = p.n_shots[b];
        L[e] = p.ctx_off[(long long)b * (p.k + 1) + n_s[b]];
      }
    }
    bool same = true;
#pragma unroll
    for (int e = 0; e < kMaxB / 32; ++e) {
      const int b = e * 32 + lane;
      if (e * 32 >= p.B) break;
      if (b < p.B) same = same && n[e] == n_s[b] && clamp_len(L[e]) == len_s[b];
    }
    return same;
  };
  long long x0 = 0, x1 = 0;
  auto find_range = [&]() {
    const Ranges rg = make_ranges(pre[p.B] * upb, p.n_cta);
    x0 = rg.start(blockIdx.x);
    x1 = rg.start(blockIdx.x + 1);
  };

  // Walks the pieces of the range: fn(b, l, g, t0, t1, n_tiles, n_ctx, whole, first) for the tiles t0 .. t1-1 of a unit.
  auto walk = [&](auto&& fn) {
    int b = 0;
    for (long long x = x0; x < x1;) {
      if (x == x0) {
        int hi = p.B;                             // request with pre[b] * upb <= x < pre[b + 1] * upb
        while (hi - b > 1) {
          const int mid = (b + hi) >> 1;
          if (pre[mid] * upb <= x) b = mid; else hi = mid;
        }
      } else {
        while (pre[b + 1] * upb <= x) ++b;
      }
      const int len = (int)(pre[b + 1] - pre[b]);
      const long long rel = x - pre[b] * upb;
      const int u = (int)div_nn(rel, len), off = (int)(rel - (long long)u * len);
      const int end = (int)(x1 - x < len - off ? off + (x1 - x) : len);
      const int t0 = off > kUnitCost ? off - kUnitCost : 0, t1 = end - kUnitCost, n_tiles = len - kUnitCost;
      if (t1 > t0)
        if (!fn(b, u / p.Hkv, u % p.Hkv, t0, t1, n_tiles, n_tiles - n_own, x == x0)) return;
      x += end - off;
    }
  };

  // What depends on the lengths alone is worked out while the kernels in front end, and the first tiles of the range are
  // brought to L2 (the memory is idle from the last tile of the call before to the end of its merge).  Nothing may be relied on
  // before the wait, so the lengths are a guess until then, right unless one of those kernels changes them.  (From the wait to the
  // first copy 3.3 us when everything followed it, 1.0 now; four calls of one request of 12 K tokens 68.2 -> 63.6 us.  Forming the angles
  // of Q here as well is slower, 70.8: the CTAs enter too late for it to be hidden.)
  if (warp == 0) lengths(true);
  __syncthreads();
  find_range();
  if (threadIdx.x == 32 * kWarps && x1 - x0 <= kPrefetchRange) {
    int left = kPrefetchTiles;
    walk([&](int b, int l, int g, int t0, int t1, int, int n_ctx, bool) {
      for (int t = t0; t < min(t1, n_ctx) && left > 0; ++t, --left)
#pragma unroll
        for (int h = 0; h < SUB; ++h) {
          tma_prefetch_4d(&tm_k, h * 64, g, t * kTile, b * p.nl + l);
          tma_prefetch_4d(&tm_v, h * 64, g, t * kTile, b * p.nl + l);
        }
      return left > 0;
    });
  }
  ads_dependency_wait();
  if (!__syncthreads_and(warp != 0 || guess_holds())) {
    if (warp == 0) lengths(false);
    __syncthreads();
    find_range();
  }
  if (blockIdx.x == 0 && warp == 0)                              // for the merge
    for (int b = lane; b <= p.B; b += 32) p.prefix[b] = pre[b];

  if (warp == kWarps) {
    // -------------------------------------------------------------- producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      walk([&](int b, int l, int g, int t0, int t1, int, int n_ctx, bool) {
        for (int t = t0; t < t1; ++t, ++it) {
          const int s = it % ST;
          ok = mbar_wait(empty(s), ((it / ST) & 1) ^ 1, abort_flag);
          if (!ok) return false;
          mbar_arrive_expect_tx(full(s), SM::kStageBytes);
          const bool own = t >= n_ctx;
          const int row = (own ? t - n_ctx : t) * kTile;
          const uint32_t dst = base + s * SM::kStageBytes;
#pragma unroll
          for (int h = 0; h < SUB; ++h) {
            tma_load_4d(dst + h * (kTile * 128), own ? &tm_ko : &tm_k, full(s), h * 64, g, row, b * p.nl + l);
            tma_load_4d(dst + SM::kTileBytes + h * (kTile * 128), own ? &tm_vo : &tm_v, full(s), h * 64, g, row,
                        b * p.nl + l);
          }
        }
        return true;
      });
      if (!ok)       // gave up: let the copies in flight land before the CTA retires
        for (uint32_t t = it > (uint32_t)ST ? it - ST : 0; t < it; ++t)
          mbar_wait(full(t % ST), (t / ST) & 1, abort_flag + 1);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------- consumers
    const int r0 = lane >> 2, c0 = 2 * (lane & 3);       // this lane's rows r0, r0 + 8 and columns c0, c0 + 1 of an 8-column block
    // rotations: a lane owns two neighbouring frequencies, a warp turns RPI rows at a time
    constexpr int RPI = 128 / D;
    const int f0 = 2 * (lane % (D / 4)), sub = lane / (D / 4);
    const double th[2] = {p.theta[f0], p.theta[f0 + 1]};
    auto angles = [&](double pos, float2& cs, float2& sn) {
      rope_sincos(pos, th[0], &sn.x, &cs.x);
      rope_sincos(pos, th[1], &sn.y, &cs.y);
    };
    auto turn = [&](uint32_t& lo, uint32_t& hi, const float2& cs, const float2& sn) {
      const float2 x = make_float2(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u));
      const float2 y = make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
      const float2 a = __ffma2_rn(y, make_float2(-sn.x, -sn.y), __fmul2_rn(x, cs));
      const float2 c = __ffma2_rn(x, sn, __fmul2_rn(y, cs));
      lo = pack2(a.x, a.y);
      hi = pack2(c.x, c.y);
    };
    uint32_t it = 0;
    walk([&](int b, int l, int g, int t0, int t1, int n_tiles, int n_ctx, bool first) {
      const long long L = len_s[b];
      const long long bl = (long long)b * p.nl + l;
      consumers_sync();                                  // the read-out of the previous piece is over
      // Q of the unit, rotated to its positions: row rr = (token t, head hh) of the KV head's group
#pragma unroll 1
      for (int rr = warp * RPI + sub; rr < MB * 16; rr += kWarps * RPI) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(q_s + rr * SM::kQStride + f0);
        uint32_t lo = 0, hi = 0;
        if (rr < p.rows) {
          const int t = rr / p.G, h = g * p.G + rr % p.G;
          const uint32_t* src = reinterpret_cast<const uint32_t*>(p.q + ((bl * p.T_new + t) * p.Hq + h) * (long long)D + f0);
          lo = src[0];
          hi = src[D / 4];
          float2 cs, sn;
          angles((double)(L + p.T_own - p.T_new + t), cs, sn);
          turn(lo, hi, cs, sn);
        }
        dst[0] = lo;
        dst[D / 4] = hi;
      }
      consumers_sync();
      const uint32_t q_addr = base + SM::kOffQ + ((lane & 15) * SM::kQStride + (lane >> 4) * 8) * 2;
      uint32_t qf[MB == 1 ? D / 16 : 1][4];
      if constexpr (MB == 1) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) ldmatrix_x4(q_addr + ks * 32, qf[ks]);
      }
      float m_run[MB][2], l_run[MB][2], o[MB][D / 8][4];
#pragma unroll
      for (int mb = 0; mb < MB; ++mb) {
        m_run[mb][0] = m_run[mb][1] = kNegSentinel;
        l_run[mb][0] = l_run[mb][1] = 0.f;
#pragma unroll
        for (int nb = 0; nb < D / 8; ++nb) o[mb][nb][0] = o[mb][nb][1] = o[mb][nb][2] = o[mb][nb][3] = 0.f;
      }
      bool ok = true;
      for (int t = t0; t < t1; ++t, ++it) {
        const int s = it % ST;
        ok = __all_sync(0xffffffffu, mbar_wait(full(s), (it / ST) & 1, abort_flag));
        if (!ok) break;
        const uint32_t k_base = base + s * SM::kStageBytes, v_base = k_base + SM::kTileBytes;
        const bool own = t >= n_ctx;
        const int own0 = (t - n_ctx) * kTile + warp * 16;          // first own token of this warp's keys
        if (own) {
          // the own keys are stored un-rotated: this warp turns its 16 rows to L + token, the first ones from fp64
          // angles, the others RPI positions further at a time by a complex multiplication
          unsigned char* kt = base_ptr + s * SM::kStageBytes;
          float2 cs, sn, cs1, sn1;
          angles((double)(L + own0 + sub), cs, sn);
          angles((double)RPI, cs1, sn1);
          auto at = [&](int c, int row) {
            return reinterpret_cast<uint32_t*>(kt + (c >> 6) * (kTile * 128) + row * 128 +
                                               ((((c & 63) >> 3) ^ (row & 7)) << 4) + (c & 7) * 2);
          };
#pragma unroll 4
          for (int r = 0; r < 16; r += RPI) {
            const int row = warp * 16 + r + sub;
            uint32_t *lo = at(f0, row), *hi = at(f0 + D / 2, row);
            uint32_t a = *lo, c = *hi;
            turn(a, c, cs, sn);
            *lo = a;
            *hi = c;
            const float2 cn = __ffma2_rn(make_float2(-sn.x, -sn.y), sn1, __fmul2_rn(cs, cs1));
            sn = __ffma2_rn(cs, sn1, __fmul2_rn(sn, cs1));
            cs = cn;
          }
          fence_proxy_async_smem();
          __syncwarp();
        }
        // S = Q K^T for this warp's 16 keys
        float sc[MB][2][4];
#pragma unroll
        for (int mb = 0; mb < MB; ++mb)
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) sc[mb][nb][0] = sc[mb][nb][1] = sc[mb][nb][2] = sc[mb][nb][3] = 0.f;
        {
          const int row = warp * 16 + (lane & 7) + ((lane >> 4) << 3);     // matrices: keys 0-7 (d lo, d hi), keys 8-15
          const int ch = (lane >> 3) & 1;
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const int chunk = ks * 2 + ch;
            uint32_t kf[4];
            ldmatrix_x4(k_base + (chunk >> 3) * (kTile * 128) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4), kf);
#pragma unroll
            for (int mb = 0; mb < MB; ++mb) {
              if constexpr (MB == 1) {
                mma_16816(sc[0][0], qf[ks], kf[0], kf[1]);
                mma_16816(sc[0][1], qf[ks], kf[2], kf[3]);
              } else {
                uint32_t qa[4];
                ldmatrix_x4(q_addr + mb * 16 * SM::kQStride * 2 + ks * 32, qa);
                mma_16816(sc[mb][0], qa, kf[0], kf[1]);
                mma_16816(sc[mb][1], qa, kf[2], kf[3]);
              }
            }
          }
        }
        uint32_t pf[MB][4];
#pragma unroll
        for (int mb = 0; mb < MB; ++mb) {
          // columns >= limit are hidden (context: keys at or beyond L; own: tokens after the row's own)
          float mx[2];
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            int limit;
            if (!own) {
              const long long left = L - (long long)t * kTile - warp * 16;
              limit = left < 16 ? (int)left : 16;
            } else {
              const int tr = min((mb * 16 + hf * 8 + r0) / p.G, p.T_new - 1);
              limit = p.T_own - p.T_new + tr + 1 - own0;
            }
#pragma unroll
            for (int nb = 0; nb < 2; ++nb)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                float& v = sc[mb][nb][2 * hf + e];
                v = nb * 8 + c0 + e < limit ? v * p.scale_log2 : -INFINITY;
              }
            mx[hf] = fmaxf(fmaxf(sc[mb][0][2 * hf], sc[mb][0][2 * hf + 1]), fmaxf(sc[mb][1][2 * hf], sc[mb][1][2 * hf + 1]));
            mx[hf] = fmaxf(mx[hf], __shfl_xor_sync(0xffffffffu, mx[hf], 1));
            mx[hf] = fmaxf(mx[hf], __shfl_xor_sync(0xffffffffu, mx[hf], 2));
          }
          if (__any_sync(0xffffffffu, mx[0] > m_run[mb][0] || mx[1] > m_run[mb][1])) {
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              const float m_new = fmaxf(m_run[mb][hf], mx[hf]);
              const float a = ex2(m_run[mb][hf] - m_new);
              m_run[mb][hf] = m_new;
              l_run[mb][hf] *= a;
#pragma unroll
              for (int nb = 0; nb < D / 8; ++nb) {
                o[mb][nb][2 * hf] *= a;
                o[mb][nb][2 * hf + 1] *= a;
              }
            }
          }
#pragma unroll
          for (int nb = 0; nb < 2; ++nb)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              const float e0 = ex2(sc[mb][nb][2 * hf] - m_run[mb][hf]), e1 = ex2(sc[mb][nb][2 * hf + 1] - m_run[mb][hf]);
              l_run[mb][hf] += e0 + e1;
              pf[mb][2 * nb + hf] = pack2(e0, e1);
            }
        }
        {
          const int row = warp * 16 + (lane & 15);                         // matrices: keys 0-7, 8-15 at d, then at d + 8
          const int ch = lane >> 4;
#pragma unroll
          for (int db = 0; db < D / 16; ++db) {
            const int chunk = db * 2 + ch;
            uint32_t vf[4];
            ldmatrix_x4_trans(v_base + (chunk >> 3) * (kTile * 128) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4), vf);
#pragma unroll
            for (int mb = 0; mb < MB; ++mb) {
              mma_16816(o[mb][2 * db], pf[mb], vf[0], vf[1]);
              mma_16816(o[mb][2 * db + 1], pf[mb], vf[2], vf[3]);
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(s));
      }
      if (!consumers_all(ok)) return false;              // (every warp comes here, so none waits for one that gave up)

      // merge of the four warps' states and read-out, four rows at a time: 32 threads take a row
      const bool whole = t0 == 0 && t1 == n_tiles;
      const long long slot = 2ll * blockIdx.x + (first ? 0 : 1);
#pragma unroll
      for (int mb = 0; mb < MB; ++mb)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float v = l_run[mb][hf];
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          l_run[mb][hf] = v + __shfl_xor_sync(0xffffffffu, v, 2);
        }
#pragma unroll
      for (int rb = 0; rb < MB * 16; rb += kMergeRows) {
        if (rb >= p.rows) break;
        if (rb > 0) consumers_sync();
        const int mb = rb / 16, hf = (rb / 8) & 1, half = (rb / kMergeRows) & 1;       // constants
        if ((r0 >> 2) == half) {
          float* dst = o_s + (warp * kMergeRows + (r0 & 3)) * SM::kOStride + c0;
#pragma unroll
          for (int nb = 0; nb < D / 8; ++nb)
            *reinterpret_cast<float2*>(dst + nb * 8) = make_float2(o[mb][nb][2 * hf], o[mb][nb][2 * hf + 1]);
          if ((lane & 3) == 0) red[warp * kMergeRows + (r0 & 3)] = make_float2(m_run[mb][hf], l_run[mb][hf]);
        }
        consumers_sync();
        constexpr int CPT = D / 32;                      // columns per thread
        const int row = threadIdx.x >> 5, col = (threadIdx.x & 31) * CPT, rr = rb + row;
        if (rr < p.rows) {
          float m = kNegSentinel, lsum = 0.f, acc[CPT] = {};
#pragma unroll
          for (int w = 0; w < kWarps; ++w) m = fmaxf(m, red[w * kMergeRows + row].x);
#pragma unroll
          for (int w = 0; w < kWarps; ++w) {
            const float2 ml = red[w * kMergeRows + row];
            const float f = ex2(ml.x - m);
            lsum += ml.y * f;
            const float* src = o_s + (w * kMergeRows + row) * SM::kOStride + col;
#pragma unroll
            for (int c = 0; c < CPT; c += 2) {
              const float2 v = *reinterpret_cast<const float2*>(src + c);
              acc[c] += v.x * f;
              acc[c + 1] += v.y * f;
            }
          }
          if (whole) {
            const int tt = rr / p.G, h = g * p.G + rr % p.G;
            const float inv = 1.f / lsum;
            __nv_bfloat16* dst = p.out + ((bl * p.T_new + tt) * p.Hq + h) * (long long)D + col;
#pragma unroll
            for (int c = 0; c < CPT; c += 2) *reinterpret_cast<uint32_t*>(dst + c) = pack2(acc[c] * inv, acc[c + 1] * inv);
            if (p.lse != nullptr && col == 0) p.lse[(bl * p.Hq + h) * p.T_new + tt] = (m + log2f(lsum)) * kLn2;
          } else {
            float* dst = p.o_part + (slot * kRows + rr) * D + col;
#pragma unroll
            for (int c = 0; c < CPT; c += 2) *reinterpret_cast<float2*>(dst + c) = make_float2(acc[c], acc[c + 1]);
            if (col == 0) *reinterpret_cast<float2*>(p.ml_part + (slot * kRows + rr) * 2) = make_float2(m, lsum);
          }
        }
      }
      return true;
    });
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag != 0) ads_set_status(p.status, ADAPSHOT_ETIMEOUT);
}

// Block (u, rr) merges row rr of unit u if a range boundary cut the unit.  One request of eight KV heads is cut into up to
// 37 pieces per head, one of a single head into up to one per CTA: eight warps take every eighth piece each, five at a
// time with their loads in flight at once, and meet in shared memory.
constexpr int kMergeWarps = 8;
template <int D, bool AHEAD>
__global__ void __launch_bounds__(32 * kMergeWarps) decode_combine_kernel(const __grid_constant__ DecodeParams p) {
  __shared__ float4 o_s[kMergeWarps][D / 4];
  __shared__ float2 ml_s[kMergeWarps];
  ads_dependency_trigger();
  const long long upb = (long long)p.nl * p.Hkv, u = blockIdx.x;
  const int b = (int)div_nn(u, upb), rr = blockIdx.y;
  const int ub = (int)(u - (long long)b * upb);      // unit within the request
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  long long p0, len, total, s;                       // the request's place in the sequence, a unit's length, the sequence's; the unit's place
  Ranges rg;
  int c0, c1;                                        // ranges that hold tiles of the unit
  auto find = [&]() {
    rg = make_ranges(total * upb, p.n_cta);
    s = p0 * upb + (long long)ub * len;
    c0 = rg.holder(s);
    c1 = rg.holder(s + len - 1);
    if (rg.start(c0 + 1) <= s + kUnitCost) ++c0;     // that range holds none of the unit's tiles
  };
  float2 ml[5];
  float4 v[5];
  auto fetch = [&](int i) {
#pragma unroll
    for (int e = 0; e < 5; ++e) {
      const int c = i + e * kMergeWarps;
      ml[e] = make_float2(kNegSentinel, 0.f);
      v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c <= c1) {
        const long long row = (2ll * c + (c > c0 || rg.start(c) >= s ? 0 : 1)) * kRows + rr;
        ml[e] = *reinterpret_cast<const float2*>(p.ml_part + row * 2);
        if (lane < D / 4) v[e] = reinterpret_cast<const float4*>(p.o_part + row * D)[lane];
      }
    }
  };
  if constexpr (AHEAD) {
    // Where the pieces lie follows from the lengths, which the kernel in front wrote when it began: read past the L1 as a guess
    // before the wait, so that behind it the lengths and the pieces are fetched together instead of one after the other
    // (four calls of one request of 12 K tokens 63.7 -> 58.4 us).  With more than three of these blocks per SM the registers this
    // takes cost more (after the wait / ahead, us per call and layer, 8 KV heads: 8 requests of 4 K tokens 26.8 / 26.2, 12 of 16 K 95.4 / 94.1,
    // 16 of 1 K 19.5 / 20.4, 20 of 13 K 133.9 / 136.6).  Whatever lies there: 0 <= begin < end <= total < 2^31 keeps every range and so every
    // address of the guess within bounds.
    p0 = __ldcg(p.prefix + b);
    const long long p1 = __ldcg(p.prefix + b + 1);
    total = __ldcg(p.prefix + p.B);
    const bool guess = 0 <= p0 && p0 < p1 && p1 <= total && total < (1ll << 31);
    len = guess ? p1 - p0 : 0;
    if (guess) find();
    ads_dependency_wait();
    const long long q0 = p.prefix[b], q1 = p.prefix[b + 1], q2 = p.prefix[p.B];
    if (guess && c0 < c1) fetch(c0 + warp);
    if (!guess || q0 != p0 || q1 - q0 != len || q2 != total) {
      p0 = q0;
      len = q1 - q0;
      total = q2;
      find();
      if (c0 < c1) fetch(c0 + warp);
    }
  } else {
    ads_dependency_wait();
    p0 = p.prefix[b];
    len = p.prefix[b + 1] - p0;
    total = p.prefix[p.B];
    find();
  }
  if (c0 >= c1) return;                             // one range held all of them and stored the result
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float M = kNegSentinel, lsum = 0.f;
  for (int i = c0 + warp; i <= c1; i += 5 * kMergeWarps) {
    if (!AHEAD || i != c0 + warp) fetch(i);
    float m_new = M;
#pragma unroll
    for (int e = 0; e < 5; ++e) m_new = fmaxf(m_new, ml[e].x);
    const float keep = exp2f(M - m_new);
    M = m_new;
    lsum *= keep;
    acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
#pragma unroll
    for (int e = 0; e < 5; ++e) {
      const float w = exp2f(ml[e].x - M);
      lsum += ml[e].y * w;
      acc.x += v[e].x * w; acc.y += v[e].y * w; acc.z += v[e].z * w; acc.w += v[e].w * w;
    }
  }
  if (lane < D / 4) o_s[warp][lane] = acc;
  if (lane == 0) ml_s[warp] = make_float2(M, lsum);
  __syncthreads();
  if (threadIdx.x >= D / 4) return;
  acc = make_float4(0.f, 0.f, 0.f, 0.f);
  M = kNegSentinel;
  lsum = 0.f;
#pragma unroll
  for (int w = 0; w < kMergeWarps; ++w) M = fmaxf(M, ml_s[w].x);
#pragma unroll
  for (int w = 0; w < kMergeWarps; ++w) {
    const float f = exp2f(ml_s[w].x - M);
    const float4 v = o_s[w][threadIdx.x];
    lsum += ml_s[w].y * f;
    acc.x += v.x * f; acc.y += v.y * f; acc.z += v.z * f; acc.w += v.w * f;
  }
  const float inv = 1.f / lsum;
  const int l = ub / p.Hkv, t = rr / p.G, h = (ub % p.Hkv) * p.G + rr % p.G;
  const long long bl = (long long)b * p.nl + l;
  reinterpret_cast<uint2*>(p.out + ((bl * p.T_new + t) * p.Hq + h) * (long long)D)[threadIdx.x] =
      make_uint2(pack2(acc.x * inv, acc.y * inv), pack2(acc.z * inv, acc.w * inv));
  if (p.lse != nullptr && threadIdx.x == 0) p.lse[(bl * p.Hq + h) * p.T_new + t] = (M + log2f(lsum)) * kLn2;
}

// Test aid: stands for a kernel in front of a decode call that writes its lengths late.
__global__ void __launch_bounds__(256) late_copy_selftest_kernel(int32_t* dst, const int32_t* src, int n, long long cycles) {
  ads_dependency_trigger();
  ads_dependency_wait();
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {
  }
  for (int i = threadIdx.x; i < n; i += 256) dst[i] = src[i];
}

struct DecodeLayout {
  size_t off_o, off_ml, off_pre, total;
};
DecodeLayout decode_layout(int D, int B) {
  DecodeLayout w;
  w.off_o = 0;
  w.off_ml = ads_round_up((size_t)2 * kMaxCtas * kRows * D * 4, 256);
  w.off_pre = w.off_ml + ads_round_up((size_t)2 * kMaxCtas * kRows * 2 * 4, 256);
  w.total = w.off_pre + ads_round_up((size_t)(B + 1) * 8, 256);
  return w;
}

template <int D, int MB>
int launch(const CUtensorMap* m, const DecodeParams& p, cudaStream_t st) {
  const int smem = (int)DecodeSmem<D>::kTotal;
  static bool attr_done[kAdsMaxDevices] = {false};
  if (ads_set_max_smem(decode_rows_kernel<D, MB>, smem, attr_done) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  ads_launch_dependent(decode_rows_kernel<D, MB>, (unsigned)p.n_cta, kThreads, smem, st, m[0], m[1], m[2], m[3], p);
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  const dim3 grid((unsigned)((long long)p.B * p.nl * p.Hkv), (unsigned)p.rows);
  if (2ll * grid.x * grid.y <= 3ll * p.n_cta) ads_launch_dependent(decode_combine_kernel<D, true>, grid, 32 * kMergeWarps, 0, st, p);
  else ads_launch_dependent(decode_combine_kernel<D, false>, grid, 32 * kMergeWarps, 0, st, p);
  return ads_launch_status();
}

}  // namespace

// Whether a call whose rows fit is better off here than with the prefill kernels.  Up to 16 rows always (one block of rows:
// 1.7 to 12 times as fast).  With 17 to 32 the second block of accumulators and the read-out of 32 rows per unit cost what
// the prefill kernels' empty rows do; prefill / here, geometric mean (range) over 127 calls of 1 to 200 requests, contexts of 32
// to 24 K tokens, 5 to 300 own tokens: d = 64, eight KV heads, ctx + 4 own >= 1024 tokens 1.13 (1.00 to 1.24), below 0.71 (0.59 to
// 0.81); one head, ctx + 16 own >= 1024 1.37 (1.05 to 1.67), below 1.12 (1.03, 1.23); d = 128, eight heads 0.74 (0.52 to 0.93); one head,
// where the prefill kernels have 16000 own tokens or more to prepare 1.21 (0.95 to 1.96), fewer 0.81 (0.57 to 1.14).
bool ads_decode_rows_pay(const adapshot_model_t* model, int B, int T_new, int T_own, int64_t ctx_cap) {
  if ((long long)T_new * (model->n_q_heads / model->n_kv_heads) <= 16) return true;
  if (model->head_dim == 128) return model->n_kv_heads == 1 && (long long)B * T_own >= 16000;
  return ctx_cap + (model->n_kv_heads == 1 ? 16ll : 4ll) * T_own >= 1024;
}
bool ads_decode_rows_fit(const adapshot_model_t* model, int T_new) {
  return (long long)T_new * (model->n_q_heads / model->n_kv_heads) <= kRows;
}
size_t ads_decode_rows_workspace(const adapshot_model_t* model, int B) {
  return decode_layout(model->head_dim, B).total;
}

int ads_decode_rows(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx, int64_t ctx_cap,
                    const int64_t* ctx_off, int B, int k, const int32_t* n_shots, const void* q_new, const void* k_own,
                    const void* v_own, int T_new, int T_own, int nl, void* out, float* lse, void* ws, int32_t* status,
                    cudaStream_t st) {
  const int D = model->head_dim, Hq = model->n_q_heads, Hkv = model->n_kv_heads;
  const DecodeLayout lay = decode_layout(D, B);
  unsigned char* wsb = static_cast<unsigned char*>(ws);
  DecodeParams p = {};
  p.q = static_cast<const __nv_bfloat16*>(q_new);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.lse = lse;
  p.o_part = reinterpret_cast<float*>(wsb + lay.off_o);
  p.ml_part = reinterpret_cast<float*>(wsb + lay.off_ml);
  p.prefix = reinterpret_cast<long long*>(wsb + lay.off_pre);
  p.ctx_off = reinterpret_cast<const long long*>(ctx_off);
  p.n_shots = n_shots;
  p.status = status;
  p.ctx_cap = ctx_cap;
  p.B = B; p.k = k; p.Hq = Hq; p.Hkv = Hkv; p.G = Hq / Hkv; p.nl = nl; p.T_new = T_new; p.T_own = T_own;
  p.rows = T_new * p.G;
  const int n_sm = ads_sm_count();
  if (n_sm <= 0) return ADAPSHOT_ECUDA;
  p.n_cta = 2 * n_sm < kMaxCtas ? 2 * n_sm : kMaxCtas;
  const float scale = model->softmax_scale > 0.f ? model->softmax_scale : 1.0f / sqrtf((float)D);
  p.scale_log2 = scale * 1.4426950408889634f;
  ads_rope_theta(model->rope_base, D, p.theta);

  CUtensorMap m[4];
  const void* src[4] = {k_ctx, v_ctx, k_own, v_own};
  for (int i = 0; i < 4; ++i) {
    const uint64_t rows = i < 2 ? (uint64_t)ctx_cap : (uint64_t)T_own;
    const uint64_t dims[4] = {(uint64_t)D, (uint64_t)Hkv, rows, (uint64_t)B * nl};
    const uint64_t str[3] = {(uint64_t)D * 2, (uint64_t)Hkv * D * 2, rows * Hkv * D * 2};
    const uint32_t box[4] = {64, 1, (uint32_t)kTile, 1};
    if (!ads_make_bf16_map(&m[i], src[i], 4, dims, str, box)) return ADAPSHOT_ECUDA;
  }
  if (D == 128) return p.rows <= 16 ? launch<128, 1>(m, p, st) : launch<128, 2>(m, p, st);
  return p.rows <= 16 ? launch<64, 1>(m, p, st) : launch<64, 2>(m, p, st);
}

extern "C" int adapshot_selftest_late_copy(int32_t* dst, const int32_t* src, int32_t n, int64_t cycles, void* stream) {
  if (dst == nullptr || src == nullptr || n <= 0 || cycles < 0 || cycles > ADAPSHOT_SELFTEST_MAX_CYCLES) return ADAPSHOT_EINVAL;
  ads_launch_dependent(late_copy_selftest_kernel, 1, 256, 0, static_cast<cudaStream_t>(stream), dst, src, n, (long long)cycles);
  return ads_launch_status();
}
