// Attention-based relevance ranking (paper Sec. 4.2, Eq. 5 and the ranking sentence after it): the
// query's Q at a representative layer against the cached K of every shot of the pool.  Eq. 5 as
// printed normalises over one shot's own tokens, which makes every shot's mean score 1 / T_i; the
// reading taken here is ONE softmax per query token and head over the keys of the whole pool, a
// shot's relevance being the attention mass that falls on its tokens, averaged over query tokens
// and heads (optionally divided by T_i).  Q and K enter as stored; 1/sqrt(d) scaling as in Eq. 5.
//
// On the tensor cores (tcgen05, S in TMEM, tiles staged by TMA), in one pass over the pool's K of that layer.  The
// normaliser of a row is only known after all keys have been seen, so the pass leaves, for every query row and shot,
// the log2 of the row's un-normalised mass on the shot, relative to the row's first maximum in that range of keys:
//   pass    S = Q K^T, one thread per query row (TMEM lane): running maximum, exponentials, and their sum over
//           every shot of the CTA's range of keys, written as maximum - first maximum + log2(sum) at the shot's end;
//   merge   the ranges' maxima and sums -> what is left to add to a range's pieces: its first maximum - log2-sum-exp of
//           the row;
//   reduce  mass of a shot = sum over rows of 2^(its piece + the row's share), one to eight warps per shot.
// (Both are small where the mass is, however large the scores are. As maximum + log2(sum) every piece carried the rounding of
// the maximum, each shot its own: 2.5e-5 of a shot's mass at logits of 2048, now 3e-6 at most.)
// What lies between the steps is 4 bytes per row and shot; the rows are taken in batches (of M tiles, and of KV heads where
// one tile is too much) that keep it below kPieceBytes.
// Where shots are short (fewer than kShortShot tokens on average) a piece per row and shot costs more than seeing the keys
// again: there a second pass, with the normalisers known, takes the places of the pieces and of their reduction.  Its score
// tiles are the other way round, a thread per key, so that a key's masses add up over the rows in its thread:
//   pass 1  running maximum and sum of every row;  merge  -> maximum and 1 / sum;
//   pass 2  mass of a key and KV head = sum over the query's rows of 2^(score - maximum) / sum;
//   keys    mass of a shot = sum over its keys and the heads.
// One pass / two, 32 / 8 heads, d = 128, 8 queries x 256 tokens: 2.5 tokens per shot (30000 shots) 12061 / 3295 us, 8 tokens
// (4000) 2248 / 1472, 12 tokens (2000) 1397 / 1279, 24 tokens (3000) 2662 / 3123; one query of 8 tokens 224 / 130, 67 / 64,
// 48 / 53, 74 / 116.  2 queries x 128 tokens over 328 K keys in shots of 160 tokens: 912 us with one pass, 1842 with two (the
// form before the pieces).
// The scores then go through the same top-k as the embedding selector (ties -> lower shot id).
#include <float.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.cuh"

namespace {

using namespace sm100;

constexpr int kTile = 128;            // query rows per M tile, keys per tile
constexpr int kGroups = 4;            // consumer groups of a CTA: a warpgroup each, one thread per row (TMEM lane) of its score tile
constexpr int kRelThreads = 128 * (kGroups + 1);      // warp 0 TMA, warp 1 MMA; consumers from warp 4 on
constexpr int kSmemTiles = 6;         // 128-row tiles in shared memory: the Q tiles, and K tiles in the rest
// Registers per thread of the first warpgroup and of the consumers; together what 640 threads are launched with, 5 x 96.
constexpr int kRelRegsIssue = 64, kRelRegsConsumer = 104;
static_assert(kRelRegsIssue + kGroups * kRelRegsConsumer <= 5 * 96, "register split");

// 2^x by the hardware approximation (one MUFU operation, relative error about 2^-22; 2^-inf = 0)
__device__ __forceinline__ float rel_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 2^x for a pair of scores on the FMA pipe (for x <= 0 or thereabouts; x below -125, -inf included, gives
// about 2^-125 instead of 0, which no sum here can see):
// x = n + f with n = round(x) taken from the low mantissa bits of x + 1.5 * 2^23, 2^f by the quartic on
// [-0.5, 0.5] whose largest relative error is smallest (2.6e-6; 7e-7 at f = 0, where every row's largest score lies:
// a cubic, 7.2e-5 there, made the masses of peaked rows wrong by 1.6e-5), n added to the exponent field.  The
// passes send every fourth pair here: the exponential unit (16 results per clock and SM) is what
// bounds it together with instruction issue (none there / every eighth / every fourth pair: 3 queries of 213 tokens over
// 275 K pool tokens 2136 / 2054 / 2043 us, 6 of 170 tokens over 596 K, d = 64, 7301 / 6852 / 6690).
__device__ __forceinline__ float2 rel_ex2_poly2(float2 x) {
  const float kMagic = 12582912.f;
  x.x = fmaxf(x.x, -125.f);      // keeps the exponent field of the result positive
  x.y = fmaxf(x.y, -125.f);
  const float2 t = __fadd2_rn(x, make_float2(kMagic, kMagic));
  const float2 n = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
  const float2 f = __fadd2_rn(x, make_float2(-n.x, -n.y));
  float2 p = __ffma2_rn(make_float2(0.009570102207f, 0.009570102207f), f, make_float2(0.05591785908f, 0.05591785908f));
  p = __ffma2_rn(p, f, make_float2(0.2402474433f, 0.2402474433f));
  p = __ffma2_rn(p, f, make_float2(0.6931217909f, 0.6931217909f));
  p = __ffma2_rn(p, f, make_float2(0.9999992847f, 0.9999992847f));
  return make_float2(__uint_as_float(__float_as_uint(p.x) + (__float_as_uint(t.x) << 23)),
                     __uint_as_float(__float_as_uint(p.y) + (__float_as_uint(t.y) << 23)));
}

// A unit is an M tile (of a query) and a KV head; units of a batch (M tiles from tile0 on, heads from head0 on) are numbered
// from 0.
struct RelParams {
  float2* norm;                 // [unit][128]: (-max, 1 / sum) of every row (two passes)
  float* key_mass;              // [query of the batch][head of the batch][n_tiles * 128] (two passes)
  float* ml_part;               // [unit][split][3][128]: max (log2 units), sum, first max; the merge replaces the last
  float* pieces;                // [unit][n_shots + splits][128]: log2 mass of row on shot i in range s - first max, at slot s + i
  const long long* shot_off;
  int32_t* status;
  long long pool_tokens;
  int Hkv, n_mt, n_shots, layer, tile0;     // tile0: first of the batch's M tiles (b * n_mt + mt)
  int head0, n_heads;           // KV heads of the batch
  int n_tiles, splits, tiles_per_split;
  int n_m, m_per_cta;           // M tiles of the batch; how many of them share a CTA's K tiles (1, 2 or 4)
  float scale_log2;
};

// q [B][Tq][Hq][D] -> q_pack [B][Hkv][n_mt * 128][D]: row m = t * G + hh of kv head g holds query
// head g * G + hh of token t; rows beyond T_q * G are zero.
template <int D>
__global__ void __launch_bounds__(256) rel_pack_q_kernel(const __nv_bfloat16* __restrict__ q,
                                                         __nv_bfloat16* __restrict__ q_pack, int B, int Tq, int Hq,
                                                         int Hkv, int rows_pad) {
  constexpr int VPR = D / 8;                         // 16-byte vectors per row
  ads_dependency_wait();
  const int G = Hq / Hkv;
  const long long n = (long long)B * Hkv * rows_pad * VPR;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int v = (int)(i % VPR);
  const long long row_g = i / VPR;
  const int m = (int)(row_g % rows_pad);
  const int g = (int)((row_g / rows_pad) % Hkv);
  const int b = (int)(row_g / ((long long)rows_pad * Hkv));
  uint4 val = make_uint4(0, 0, 0, 0);
  if (m < Tq * G) {
    const int t = m / G, hh = m % G;
    val = reinterpret_cast<const uint4*>(q)[(((long long)b * Tq + t) * Hq + g * G + hh) * VPR + v];
  }
  reinterpret_cast<uint4*>(q_pack)[i] = val;
}

enum RelBar { kRQFull = 0, kRKFull = 1, kRKEmpty = 6, kRSFull = 11, kRSEmpty = 15, kRDrain = 19, kRNumBars = 20 };

template <int D>
struct RelSmem {
  static constexpr uint32_t kTileBytes = (D / 64) * 16384u;
  static constexpr uint32_t kOffBar = kSmemTiles * kTileBytes;
  static constexpr uint32_t kTotal = kOffBar + 256 + 1024;      // + alignment slack
};

// grid (groups of M tiles, groups of key ranges, KV heads).  The four consumer groups of a CTA take m_per_cta M tiles times
// 4 / m_per_cta key ranges: group x has M tile x % m_per_cta and range x / m_per_cta.  M tiles of a CTA share
// every K tile; where there are few of them the ranges keep all groups busy.  CTAs that differ in their M tiles only
// walk the same key tiles at the same time, so the pool's K layer is read from DRAM about once.
// Bound by the exponential unit (128 x 128 results per score tile, 16 per clock and SM) and, where shots end, by
// instruction issue: sixteen consumer warps keep both busy under each other's latencies.  (Two CTAs per SM with one M
// tile and four consumer warps each: 1000 us for 2 queries x 128 tokens, 328 K pool tokens; 790 us now, the exponential unit
// and the issue slots both two thirds busy.)
//
// STEP: what is done with the scores.  In kMasses the operands change places: a CTA keeps up to four K tiles (m_per_cta), a
// consumer group's rows are the keys of one of them, and the M tiles of the batch stream by.
enum RelStep { kPieces, kNormalisers, kMasses };
template <int D, int STEP>
__global__ void __launch_bounds__(kRelThreads, 1)
rel_pass_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                const __grid_constant__ RelParams p) {
  using SM = RelSmem<D>;
  constexpr int SUB = D / 64;
  constexpr uint32_t kTileBytes = SM::kTileBytes;
  constexpr uint32_t kIdesc = idesc_bf16_f32(kTile, kTile, 0);
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_raw + (base - raw_addr);
  const uint32_t bar0 = base + SM::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * i; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + SM::kOffBar + 8 * kRNumBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + SM::kOffBar + 8 * kRNumBars + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = p.head0 + blockIdx.z;
  const int m0 = blockIdx.x * p.m_per_cta;          // tiles that stay: M tiles of this CTA (kMasses: K tiles)
  const int n_m = min(p.m_per_cta, (STEP == kMasses ? p.n_tiles : p.n_m) - m0);
  const int s0 = blockIdx.y * (kGroups / p.m_per_cta);                                // its ranges
  const int n_s = STEP == kMasses ? 1 : min(kGroups / p.m_per_cta, p.splits - s0);
  const int m_stream = blockIdx.y * p.tiles_per_split;                               // kMasses: first M tile that streams by
  const int stages = kSmemTiles - p.m_per_cta;
  const uint32_t k_base = base + p.m_per_cta * kTileBytes;
  // tiles of range s0 + j: the last range of a call may be shorter than the others
  auto range_tiles = [&](int j) {
    if constexpr (STEP == kMasses) return min(p.n_m - m_stream, p.tiles_per_split);
    return max(0, min(p.n_tiles, (s0 + j + 1) * p.tiles_per_split) - (s0 + j) * p.tiles_per_split);
  };
  const int n_it = range_tiles(0);

  if (threadIdx.x == 32) {
    mbar_init(bar(kRQFull), 1);
    for (int i = 0; i < stages; ++i) {
      mbar_init(bar(kRKFull + i), 1);
      mbar_init(bar(kRKEmpty + i), 1);
    }
    for (int i = 0; i < kGroups; ++i) {
      mbar_init(bar(kRSFull + i), 1);
      mbar_init(bar(kRSEmpty + i), 128);
    }
    mbar_init(bar(kRDrain), 1);
    abort_flag[0] = 0;
    abort_flag[1] = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  ads_dependency_wait();

  auto role_tma = [&]() {
    if (lane == 0) {
      tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k);
      mbar_arrive_expect_tx(bar(kRQFull), n_m * kTileBytes);
      auto load_rows = [&](uint32_t dst, uint32_t full, int m) {         // M tile m of the batch
        const int b = (p.tile0 + m) / p.n_mt, mt = (p.tile0 + m) % p.n_mt;
#pragma unroll
        for (int s = 0; s < SUB; ++s) tma_load_3d(dst + s * 16384u, &tm_q, full, s * 64, mt * kTile, b * p.Hkv + g);
      };
      auto load_keys = [&](uint32_t dst, uint32_t full, int tile) {
#pragma unroll
        for (int s = 0; s < SUB; ++s) tma_load_4d(dst + s * 16384u, &tm_k, full, s * 64, g, tile * kTile, p.layer);
      };
      for (int m = 0; m < n_m; ++m) {
        if constexpr (STEP == kMasses) load_keys(base + m * kTileBytes, bar(kRQFull), m0 + m);
        else load_rows(base + m * kTileBytes, bar(kRQFull), m0 + m);
      }
      bool ok = true;
      int st = 0, n = 0;
      uint32_t phase = 1;
      for (int i = 0; i < n_it && ok; ++i)
        for (int j = 0; j < n_s; ++j) {
          if (i >= range_tiles(j)) continue;
          ok = mbar_wait(bar(kRKEmpty + st), phase, abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar(kRKFull + st), kTileBytes);
          if constexpr (STEP == kMasses) load_rows(k_base + st * kTileBytes, bar(kRKFull + st), m_stream + i);
          else load_keys(k_base + st * kTileBytes, bar(kRKFull + st), (s0 + j) * p.tiles_per_split + i);
          ++n;
          if (++st == stages) { st = 0; phase ^= 1; }
        }
      if (!ok) {      // gave up: let the copies in flight land before the CTA retires
        mbar_wait(bar(kRQFull), 0, abort_flag + 1);
        for (int t = max(0, n - stages); t < n; ++t)
          mbar_wait(bar(kRKFull + t % stages), (t / stages) & 1, abort_flag + 1);
      }
    }
    __syncwarp();
  };
  auto role_mma = [&]() {
    if (lane == 0) {
      constexpr uint32_t kHi = smem_desc_hi_sw128(1024);
      const uint32_t q_lo0 = smem_desc_lo(base, 16), k_lo0 = smem_desc_lo(k_base, 16);
      bool ok = mbar_wait(bar(kRQFull), 0, abort_flag);
      int st = 0;
      uint32_t phase = 0;
      for (int i = 0; i < n_it && ok; ++i)
        for (int j = 0; j < n_s && ok; ++j) {
          if (i >= range_tiles(j)) continue;
          ok = mbar_wait(bar(kRKFull + st), phase, abort_flag);
          const uint32_t k_lo = k_lo0 + st * (kTileBytes >> 4);
          for (int m = 0; m < n_m && ok; ++m) {
            const int x = j * p.m_per_cta + m;
            ok = mbar_wait(bar(kRSEmpty + x), (i & 1) ^ 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t q_lo = q_lo0 + m * (kTileBytes >> 4), d = tmem_base + x * kTile;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint32_t o = ((ks / 4) * 16384u + (ks % 4) * 32u) >> 4;
              umma_ss_lohi(d, q_lo + o, kHi, k_lo + o, kHi, kIdesc, ks > 0 ? 1u : 0u);
            }
            umma_commit(bar(kRSFull + x));
          }
          if (!ok) break;
          umma_commit(bar(kRKEmpty + st));
          if (++st == stages) { st = 0; phase ^= 1; }
        }
      if (!ok) {      // gave up: the UMMAs already issued must be done before the tensor memory is freed
        umma_commit(bar(kRDrain));
        mbar_wait(bar(kRDrain), 0, abort_flag + 1);
      }
    }
    __syncwarp();
  };
  auto role_masses = [&]() {
    const int x = (warp >> 2) - 1, quarter = warp & 3, r = quarter * 32 + lane;      // TMEM lane: key of the tile
    if (x >= n_m) return;
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    float* out = p.key_mass + (long long)blockIdx.z * p.n_tiles * kTile + (long long)(m0 + x) * kTile + r;
    const long long per_query = (long long)p.n_heads * p.n_tiles * kTile;
    double sum = 0.0;
    for (int i = 0; i < n_it; ++i) {
      if (!__all_sync(0xffffffffu, mbar_wait(bar(kRSFull + x), i & 1, abort_flag))) return;
      tc_fence_after();
      const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
      float2 part[2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        constexpr int kCols = kTile / 2;
        float s[kCols];
        tmem_ld2x32(tmem_base + lane_addr + x * kTile + half * kCols, reinterpret_cast<uint32_t*>(s));
        if (half == 1) {
          tc_fence_before();
          mbar_arrive(bar(kRSEmpty + x));
        }
        // the rows' normalisers, two rows per load, the same address in every lane
        const float4* nm = reinterpret_cast<const float4*>(p.norm + ((long long)(m_stream + i) * p.n_heads + blockIdx.z) * kTile + half * kCols);
#pragma unroll
        for (int c = 0; c < kCols; c += 2) {
          const float4 n = nm[c / 2];
          const float2 a = __ffma2_rn(make_float2(s[c], s[c + 1]), scale2, make_float2(n.x, n.z));
          const float2 e = ((c >> 1) & 3) == 3 ? rel_ex2_poly2(a) : make_float2(rel_ex2(a.x), rel_ex2(a.y));
          part[(c >> 1) & 1] = __ffma2_rn(e, make_float2(n.y, n.w), part[(c >> 1) & 1]);
        }
      }
      const float2 both = __fadd2_rn(part[0], part[1]);
      sum += (double)(both.x + both.y);
      const int tile = p.tile0 + m_stream + i;
      if ((tile + 1) % p.n_mt == 0) {                        // the query's last tile (batches and their parts hold whole queries)
        out[(long long)(tile / p.n_mt - p.tile0 / p.n_mt) * per_query] = (float)sum;
        sum = 0.0;
      }
    }
  };
  auto role_consume = [&]() {
    const int x = (warp >> 2) - 1, quarter = warp & 3;
    const int m = x % p.m_per_cta, j = x / p.m_per_cta;
    if (m >= n_m || j >= n_s) return;                       // fewer M tiles or ranges than the CTA has room for
    const int split = s0 + j, n_mine = range_tiles(j), t0 = split * p.tiles_per_split, t1 = t0 + n_mine;
    const long long unit = (long long)(m0 + m) * p.n_heads + blockIdx.z;
    const int r = quarter * 32 + lane;                      // TMEM lane: query row
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    float m_run = -1.0e30f, l_run = 0.f, acc = 0.f;         // running maximum, sum of the shots so far, of the current one
    float m_first = 0.f;                                    // the maximum of the first keys (0 where they have none)
    // the current shot and where it and the next one end (the last one with the pool); the same in every lane
    auto shot_end = [&](int i) -> long long {
      return i + 1 < p.n_shots ? p.shot_off[i + 1] : i + 1 == p.n_shots ? p.pool_tokens : (1ll << 62);
    };
    // (found by a 32-ary search of the whole warp: the steps of a binary one are a chain of cold loads)
    int shot = 0;
    for (int seg = STEP == kNormalisers ? 1 : p.n_shots; seg > 1;) {
      const int stride = (seg + 31) / 32, at = shot + lane * stride;
      const bool le = lane == 0 || (at < shot + seg && p.shot_off[at] <= (long long)t0 * kTile);
      const int first = shot + (__popc(__ballot_sync(0xffffffffu, le)) - 1) * stride;
      seg = min(stride, shot + seg - first);
      shot = first;
    }
    if (STEP == kNormalisers) shot = p.n_shots;             // (nothing ends)
    long long end = shot_end(shot), end_next = shot_end(shot + 1);
    float* piece = p.pieces + ((unit * (p.n_shots + p.splits) + split + shot) * kTile + r);
    auto flush = [&]() {                                    // the current shot is complete (in this range)
      *piece = (m_run - m_first) + __log2f(acc);
      l_run += acc;
      acc = 0.f;
      piece += kTile;
      ++shot;
      end = end_next;
      end_next = shot_end(shot + 1);
    };
    bool ok = true;
    for (int i = 0; i < n_mine; ++i) {
      ok = __all_sync(0xffffffffu, mbar_wait(bar(kRSFull + x), i & 1, abort_flag));
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        constexpr int kCols = kTile / 2;                    // (a whole row at once would not fit the registers)
        float s[kCols];
        tmem_ld2x32(tmem_base + lane_addr + x * kTile + half * kCols, reinterpret_cast<uint32_t*>(s));
        if (half == 1) {                                    // the scores are in registers: the buffer is free
          tc_fence_before();
          mbar_arrive(bar(kRSEmpty + x));
        }
        const long long key0 = (long long)(t0 + i) * kTile + half * kCols;
        if (key0 + kCols > p.pool_tokens) {        // only the pool's last tile: keys beyond it count as -inf
          const int limit = (int)max(0ll, p.pool_tokens - key0);
#pragma unroll
          for (int c = 0; c < kCols; ++c) s[c] = c < limit ? s[c] : -INFINITY;
        }
        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < kCols; c += 8) {
#pragma unroll
          for (int u = 0; u < 4; ++u) mx4[u] = fmax3(mx4[u], s[c + 2 * u], s[c + 2 * u + 1]);
        }
        const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * p.scale_log2;
        if (mx > m_run) {
          const float keep = rel_ex2(m_run - mx);
          l_run *= keep;
          acc *= keep;
          m_run = mx;
        }
        if (half == 0 && i == 0 && m_run > -1.0e29f) m_first = m_run;
        // two scores per FMA / add instruction; the exponentials themselves are one MUFU operation each
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2), neg_m2 = make_float2(-m_run, -m_run);
        float group[kCols / 8];                             // sums of 8 keys
#pragma unroll
        for (int c0 = 0; c0 < kCols; c0 += 8) {
          float2 part = make_float2(0.f, 0.f);
#pragma unroll
          for (int c = c0; c < c0 + 8; c += 2) {
            const float2 a = __ffma2_rn(make_float2(s[c], s[c + 1]), scale2, neg_m2);
            const float2 e = ((c >> 1) & 3) == 3 ? rel_ex2_poly2(a) : make_float2(rel_ex2(a.x), rel_ex2(a.y));
            s[c] = e.x;
            s[c + 1] = e.y;
            part = c == c0 ? e : __fadd2_rn(part, e);
          }
          group[c0 / 8] = part.x + part.y;
        }
        // sums per shot (the branches are the same in every lane): all keys within one shot, else group by group, the
        // keys of a group one by one only where a shot ends in it (groups of 16: 6-20 % slower at 16 to 48 tokens per shot)
        const long long left = end - key0;
        if (STEP == kNormalisers) {
          l_run += ((group[0] + group[1]) + (group[2] + group[3])) + ((group[4] + group[5]) + (group[6] + group[7]));
        } else if (left > kCols) {
          acc += ((group[0] + group[1]) + (group[2] + group[3])) + ((group[4] + group[5]) + (group[6] + group[7]));
        } else {
          int ce = (int)left;                               // columns left of the current shot
#pragma unroll
          for (int c0 = 0; c0 < kCols; c0 += 8) {
            if (ce > c0 + 8) {
              acc += group[c0 / 8];
            } else {
              int from = c0;
              while (from < c0 + 8) {
                const int to = min(ce, c0 + 8);
                float sum[2] = {0.f, 0.f};
#pragma unroll
                for (int c = 0; c < 8; ++c) sum[c & 1] += c0 + c >= from && c0 + c < to ? s[c0 + c] : 0.f;
                acc += sum[0] + sum[1];
                if (to == ce) {
                  flush();
                  ce = end - key0 > 4096 ? 4096 : (int)(end - key0);
                }
                from = to;
              }
            }
          }
        }
      }
    }
    if (ok && n_mine > 0) {
      // the shot that goes on in the next range
      if (STEP == kPieces && shot < p.n_shots && (shot == 0 || (long long)t1 * kTile > p.shot_off[shot])) flush();
      float* out = p.ml_part + (unit * p.splits + split) * 3 * kTile + r;
      out[0] = m_run;
      out[kTile] = l_run;
      out[2 * kTile] = m_first;
    }
  };

  if (warp < 4) {
    regs_lower<kRelRegsIssue>();
    if (warp == 0) role_tma();
    else if (warp == 1) role_mma();
  } else {
    regs_raise<kRelRegsConsumer>();
    if constexpr (STEP == kMasses) role_masses();
    else role_consume();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *abort_flag != 0) ads_set_status(p.status, ADAPSHOT_ETIMEOUT);
}

// What is left to add to the pieces of a row in every range: first max - log2 sum_keys 2^(s c), -inf for rows that do not exist
// (so that they add nothing).  With norm set (two passes): (-max, 1 / sum) of the row instead, 0 for the latter.  A block per
// unit: threadIdx.x is the row, every kMergeGroups-th range a thread's.  (One thread per row walked up to 256 ranges: 51 us for 4
// units of 71 ranges, 16 for 148 now.)
constexpr int kMergeGroups = 8;
__global__ void __launch_bounds__(kTile * kMergeGroups) rel_merge_kernel(float* __restrict__ ml_part, int splits, int n_heads,
                                                                         int tile0, int n_mt, int rows,
                                                                         float2* __restrict__ norm) {
  __shared__ float2 part[kMergeGroups][kTile];
  ads_dependency_wait();
  const long long unit = blockIdx.x;
  const int r = threadIdx.x, y = threadIdx.y;
  const int mt = (int)((tile0 + unit / n_heads) % n_mt);
  float* ml = ml_part + unit * splits * 3 * kTile + r;              // a range's figures are 3 * 128 floats
  float M = -1.0e30f, l = 0.f;
  for (int base = y; base < splits; base += 8 * kMergeGroups) {     // eight ranges' figures on their way at a time
    float m8[8], l8[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int s = base + e * kMergeGroups;
      m8[e] = s < splits ? ml[s * 3 * kTile] : -1.0e30f;
      l8[e] = s < splits ? ml[s * 3 * kTile + kTile] : 0.f;
    }
    float m_new = M;
#pragma unroll
    for (int e = 0; e < 8; ++e) m_new = fmaxf(m_new, m8[e]);
    l *= exp2f(M - m_new);
    M = m_new;
#pragma unroll
    for (int e = 0; e < 8; ++e) l += l8[e] * exp2f(m8[e] - M);
  }
  part[y][r] = make_float2(M, l);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kMergeGroups; ++i) M = fmaxf(M, part[i][r].x);
  l = 0.f;
#pragma unroll
  for (int i = 0; i < kMergeGroups; ++i) l += part[i][r].y * exp2f(part[i][r].x - M);
  const float log_l = log2f(l);
  const bool exists = mt * kTile + r < rows;
  if (norm != nullptr) {
    if (y == 0) norm[unit * kTile + r] = make_float2(-M, exists && l > 0.f ? 1.f / l : 0.f);
    return;
  }
#pragma unroll 8
  for (int s = y; s < splits; s += kMergeGroups) {
    float* first = ml + s * 3 * kTile + 2 * kTile;
    *first = !exists ? -INFINITY : l > 0.f ? (*first - M) - log_l : *first;
  }
}

// mass[b][i] (+)= sum over the batch's rows and heads of query b of 2^(piece + the row's share).  A block of eight warps takes
// 8 / `warps` shots of a query: the (M tile, head) units of the query are dealt out to a shot's warps, whose sums are added in
// their order.  (With a warp per shot a pool of 64 shots was eight blocks: 57 us for 8 M tiles of 8 heads, 9 now.)
__global__ void __launch_bounds__(256) rel_reduce_kernel(const float* __restrict__ pieces, const float* __restrict__ ml_part,
                                                         const long long* __restrict__ shot_off, int n_shots, int n_heads,
                                                         int n_mt, int tile0, int n_tiles_m, int splits,
                                                         int tiles_per_split, long long pool_tokens, int b0, int head0, int warps,
                                                         double* __restrict__ mass) {
  __shared__ double sum_s[8];
  ads_dependency_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = b0 + blockIdx.y;
  const int i = blockIdx.x * (8 / warps) + warp / warps, w = warp % warps;
  const int first = max(tile0, b * n_mt), last = min(tile0 + n_tiles_m, (b + 1) * n_mt);   // M tiles of this query
  double sum = 0.0;
  if (i < n_shots) {
    const long long o0 = i > 0 ? shot_off[i] : 0, o1 = i + 1 < n_shots ? shot_off[i + 1] : pool_tokens;
    const int s0 = (int)(o0 / kTile) / tiles_per_split, s1 = (int)((o1 - 1) / kTile) / tiles_per_split;
    const long long u0 = (long long)(first - tile0) * n_heads + w;                         // this warp's first unit, [m][head]
    const int n_u = ((last - first) * n_heads - w + warps - 1) / warps;
    const long long piece_step = (long long)warps * (n_shots + splits) * (kTile / 4), share_step = (long long)warps * splits * 3 * (kTile / 4);
    for (int s = s0; s <= s1; ++s) {
      const float4* pc = reinterpret_cast<const float4*>(pieces + (u0 * (n_shots + splits) + s + i) * kTile) + lane;
      const float4* share = reinterpret_cast<const float4*>(ml_part + ((u0 * splits + s) * 3 + 2) * kTile) + lane;
#pragma unroll 8
      for (int e = 0; e < n_u; ++e, pc += piece_step, share += share_step) {
        const float4 v = *pc, n = *share;
        const float part = (rel_ex2(v.x + n.x) + rel_ex2(v.y + n.y)) + (rel_ex2(v.z + n.z) + rel_ex2(v.w + n.w));
        sum += (double)part;
      }
    }
  }
  sum = warp_sum(sum);
  if (warps > 1) {
    if (lane == 0) sum_s[warp] = sum;
    __syncthreads();
    if (w == 0)
      for (int e = 1; e < warps; ++e) sum += sum_s[warp + e];
  }
  if (lane == 0 && w == 0 && i < n_shots) {
    double* out = mass + (long long)b * n_shots + i;
    *out = first == b * n_mt && head0 == 0 ? sum : *out + sum;
  }
}

// Two passes: mass[b][i] (+)= sum over the batch's heads of the masses of shot i's keys; grid (shots / 8, queries of the batch),
// a warp per shot.
__global__ void __launch_bounds__(256) rel_keys_kernel(const float* __restrict__ key_mass, const long long* __restrict__ shot_off,
                                                       int n_shots, int n_heads, int head0, long long keys_pad,
                                                       long long pool_tokens, int b0, double* __restrict__ mass) {
  ads_dependency_wait();
  const int lane = threadIdx.x & 31, i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n_shots) return;
  const long long o0 = i > 0 ? shot_off[i] : 0, o1 = i + 1 < n_shots ? shot_off[i + 1] : pool_tokens;
  const float* src = key_mass + (long long)blockIdx.y * n_heads * keys_pad;
  double sum = 0.0;
  if (o1 - o0 < 32) {                                // several heads' keys at a time
    const int len = (int)(o1 - o0);
    for (int e = lane; e < len * n_heads; e += 32) sum += (double)src[e / len * keys_pad + o0 + e % len];
  } else {
    for (int h = 0; h < n_heads; ++h)
      for (long long k = o0 + lane; k < o1; k += 32) sum += (double)src[h * keys_pad + k];
  }
  sum = warp_sum(sum);
  if (lane == 0) {
    double* out = mass + (long long)(b0 + blockIdx.y) * n_shots + i;
    *out = head0 == 0 ? sum : *out + sum;
  }
}

// score[b][i] = mass[b][i] / (T_q * Hq) (and / T_i with per_token); writes the sort keys.
__global__ void __launch_bounds__(256) rel_scores_kernel(const double* __restrict__ mass,
                                                         const long long* __restrict__ shot_off, int B, int n_shots,
                                                         double inv_rows, int per_token,
                                                         unsigned long long* __restrict__ keys) {
  ads_dependency_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)B * n_shots) return;
  const int shot = (int)(i % n_shots);
  double s = mass[i] * inv_rows;
  if (per_token) s /= (double)(shot_off[shot + 1] - shot_off[shot]);
  keys[i] = ads_desc_key(s);
}

constexpr size_t kPieceBytes = 256u << 20;
constexpr long long kShortShot = 12;     // tokens per shot on average below which two passes are taken
constexpr int kStartTiles = 4;          // what starting a CTA costs, in tiles (7 and 12 give the same times within 1 %)
constexpr long long kMaxRanges = 16 * 148 * kGroups;     // (unit, range) pairs of a launch that are worth having: sixteen waves

struct RelPlan {
  bool two_passes;
  int G, n_mt, rows, rows_pad, n_tiles, splits, tiles_per_split;
  int batch, heads;             // M tiles and KV heads per launch of the pass
  int m_per_cta;                // of which share a CTA
  size_t off_qpack, off_ml, off_norm, off_pieces, off_mass, off_keys, total;
};

RelPlan rel_plan(const adapshot_model_t* model, const adapshot_pool_t* pool, int B, int Tq) {
  RelPlan pl;
  const int D = model->head_dim, Hkv = model->n_kv_heads;
  pl.G = model->n_q_heads / Hkv;
  pl.rows = Tq * pl.G;
  pl.n_mt = (pl.rows + kTile - 1) / kTile;
  pl.rows_pad = pl.n_mt * kTile;
  pl.n_tiles = (int)((pool->pool_tokens + kTile - 1) / kTile);
  const int most = (pl.n_tiles + 1) / 2 < 256 ? (pl.n_tiles + 1) / 2 : 256;
  // What lies between the steps fits in batches of equal size: M tiles (two passes: whole queries), and KV heads where one of
  // them is too much.
  const long long m_tiles = (long long)B * pl.n_mt;
  pl.two_passes = pool->pool_tokens < kShortShot * pool->n_shots;
  const long long step = pl.two_passes ? pl.n_mt : 1;           // M tiles that stay together
  const long long fit_units = (long long)((kPieceBytes / (kTile * 4) - kMaxRanges) / (pl.two_passes ? (size_t)pl.n_tiles : (size_t)pool->n_shots));
  const long long fit = (fit_units / Hkv > 1 ? fit_units / Hkv : 1) * step;
  const long long n_batches = (m_tiles + fit - 1) / fit;
  pl.batch = (int)((m_tiles / step + n_batches - 1) / n_batches * step);
  pl.heads = Hkv;
  if (fit_units < Hkv) {
    const int n = (int)((Hkv + (fit_units > 1 ? fit_units : 1) - 1) / (fit_units > 1 ? fit_units : 1));
    pl.heads = (Hkv + n - 1) / n;
  }
  // M tiles per CTA: as many as share without leaving more than a seventh of the places empty
  pl.m_per_cta = 1;
  for (int m = 4; m > 1; m >>= 1)
    if ((pl.batch + m - 1) / m * m * 7 <= pl.batch * 8) {
      pl.m_per_cta = m;
      break;
    }
  // Key ranges: the CTAs run in waves of 148 (a fixed figure, so that the workspace size does not depend on the
  // device), each costs its tiles and a start; the split with the cheapest waves *
  // (tiles + kStartTiles) is taken, every range at least two key tiles.
  const long long units = (long long)pl.batch * pl.heads;
  const int per_cta = kGroups / pl.m_per_cta;                 // ranges of one CTA
  const long long ctas = (long long)((pl.batch + pl.m_per_cta - 1) / pl.m_per_cta) * pl.heads;
  int best_s = 1;
  long long best_cost = 0;
  for (int sp = 1; sp <= most && (sp == 1 || units * sp <= kMaxRanges); ++sp) {
    const long long tiles = (pl.n_tiles + sp - 1) / sp;
    const long long waves = (ctas * ((sp + per_cta - 1) / per_cta) + 147) / 148;
    const long long cost = waves * (tiles + kStartTiles);
    if (sp == 1 || cost < best_cost) {
      best_s = sp;
      best_cost = cost;
    }
  }
  pl.tiles_per_split = (pl.n_tiles + best_s - 1) / best_s;
  pl.splits = (pl.n_tiles + pl.tiles_per_split - 1) / pl.tiles_per_split;
  // The sizes are those of the largest batch and split that a call with no more rows than this one can have: a workspace
  // for the longest query takes the shorter ones, too.
  const long long most_units = (m_tiles < fit ? m_tiles : fit) * pl.heads;
  const long long all = most_units * most < kMaxRanges ? most_units * most : kMaxRanges;
  const size_t ranges = (size_t)(all > most_units ? all : most_units);
  size_t off = 0;
  pl.off_qpack = off;   off += ads_round_up((size_t)B * Hkv * pl.rows_pad * D * 2, 256);
  pl.off_ml = off;      off += ads_round_up(ranges * kTile * 3 * 4, 256);
  pl.off_norm = off;    off += pl.two_passes ? ads_round_up((size_t)most_units * kTile * sizeof(float2), 256) : 0;
  pl.off_pieces = off;  off += ads_round_up(
      (pl.two_passes ? (size_t)(most_units / step) * pl.n_tiles : (size_t)most_units * pool->n_shots + ranges) * kTile * 4, 256);
  pl.off_mass = off;    off += ads_round_up((size_t)B * pool->n_shots * 8, 256);
  pl.off_keys = off;    off += ads_round_up((size_t)B * pool->n_shots * 8, 256);
  pl.total = off;
  return pl;
}

bool rel_shape_ok(const adapshot_model_t* m) {
  return (m->head_dim == 64 || m->head_dim == 128) && m->n_kv_heads > 0 && m->n_q_heads > 0 &&
         m->n_q_heads % m->n_kv_heads == 0;
}

template <int D>
int rel_launch(const adapshot_model_t* model, const adapshot_pool_t* pool, int layer, const void* q, int B, int Tq,
               int k, uint32_t flags, int32_t* sel_idx, float* sel_score, const RelPlan& pl, void* ws,
               int32_t* status, cudaStream_t st) {
  const int Hq = model->n_q_heads, Hkv = model->n_kv_heads;
  unsigned char* wsb = static_cast<unsigned char*>(ws);
  __nv_bfloat16* q_pack = reinterpret_cast<__nv_bfloat16*>(wsb + pl.off_qpack);
  float* ml_part = reinterpret_cast<float*>(wsb + pl.off_ml);
  float* pieces = reinterpret_cast<float*>(wsb + pl.off_pieces);
  double* mass = reinterpret_cast<double*>(wsb + pl.off_mass);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(wsb + pl.off_keys);

  CUtensorMap tm_q, tm_k;
  {
    const uint64_t dims[3] = {(uint64_t)D, (uint64_t)pl.rows_pad, (uint64_t)B * Hkv};
    const uint64_t str[2] = {(uint64_t)D * 2, (uint64_t)pl.rows_pad * D * 2};
    const uint32_t box[3] = {64, (uint32_t)kTile, 1};
    if (!ads_make_bf16_map(&tm_q, q_pack, 3, dims, str, box)) return ADAPSHOT_ECUDA;
  }
  {
    const uint64_t dims[4] = {(uint64_t)D, (uint64_t)Hkv, (uint64_t)pool->pool_tokens, (uint64_t)model->n_layers};
    const uint64_t str[3] = {(uint64_t)D * 2, (uint64_t)Hkv * D * 2, (uint64_t)pool->pool_tokens * Hkv * D * 2};
    const uint32_t box[4] = {64, 1, (uint32_t)kTile, 1};
    if (!ads_make_bf16_map(&tm_k, pool->k, 4, dims, str, box)) return ADAPSHOT_ECUDA;
  }

  const long long n_vec = (long long)B * Hkv * pl.rows_pad * (D / 8);
  ads_launch_dependent(rel_pack_q_kernel<D>, (unsigned)((n_vec + 255) / 256), 256, 0, st,
                       static_cast<const __nv_bfloat16*>(q), q_pack, B, Tq, Hq, Hkv, pl.rows_pad);
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  const long long* shot_off = reinterpret_cast<const long long*>(pool->shot_off);
  RelParams rp;
  rp.norm = pl.two_passes ? reinterpret_cast<float2*>(wsb + pl.off_norm) : nullptr;
  rp.key_mass = pieces;
  rp.ml_part = ml_part; rp.pieces = pieces; rp.shot_off = shot_off; rp.status = status;
  rp.pool_tokens = pool->pool_tokens;
  rp.Hkv = Hkv; rp.n_mt = pl.n_mt; rp.n_shots = pool->n_shots; rp.layer = layer;
  rp.n_tiles = pl.n_tiles; rp.splits = pl.splits; rp.tiles_per_split = pl.tiles_per_split;
  const float scale = model->softmax_scale > 0.f ? model->softmax_scale : 1.0f / sqrtf((float)D);
  rp.scale_log2 = scale * 1.4426950408889634f;

  const int smem = (int)RelSmem<D>::kTotal;
  static bool attr_done[3][kAdsMaxDevices] = {{false}, {false}, {false}};
  auto launch_pass = [&](auto kernel, int which, int tiles, int ranges, int heads) -> int {
    if (ads_set_max_smem(kernel, smem, attr_done[which]) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    const int per_cta = kGroups / rp.m_per_cta;
    ads_launch_dependent(kernel, dim3((unsigned)((tiles + rp.m_per_cta - 1) / rp.m_per_cta),
                                      (unsigned)((ranges + per_cta - 1) / per_cta), (unsigned)heads),
                         kRelThreads, smem, st, tm_q, tm_k, rp);
    return ads_launch_status();
  };
  const int m_tiles = B * pl.n_mt;
  for (int t0 = 0; t0 < m_tiles; t0 += pl.batch)
    for (int h0 = 0; h0 < Hkv; h0 += pl.heads) {
      const int n = m_tiles - t0 < pl.batch ? m_tiles - t0 : pl.batch, nh = Hkv - h0 < pl.heads ? Hkv - h0 : pl.heads;
      rp.tile0 = t0;
      rp.head0 = h0;
      rp.n_heads = nh;
      rp.n_m = n;
      rp.m_per_cta = pl.m_per_cta;
      const int rc = pl.two_passes ? launch_pass(rel_pass_kernel<D, kNormalisers>, 1, n, pl.splits, nh)
                                   : launch_pass(rel_pass_kernel<D, kPieces>, 0, n, pl.splits, nh);
      if (rc != ADAPSHOT_OK) return rc;
      ads_launch_dependent(rel_merge_kernel, (unsigned)(n * nh), dim3(kTile, kMergeGroups), 0, st, ml_part, pl.splits, nh, t0,
                           pl.n_mt, pl.rows, rp.norm);
      if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
      const int b0 = t0 / pl.n_mt, b1 = (t0 + n - 1) / pl.n_mt;       // queries with rows in the batch
      if (pl.two_passes) {
        // K tiles that stay in a CTA and queries that stream by: the cheapest waves * (steps + start).  A step of four, two or
        // one K tiles takes about 4, 2.4 or 1.6 times the exponentials of one.
        const int queries = n / pl.n_mt;
        double best = 0.0;
        int per_cta = 4, parts = 1;
        for (int m = 4; m >= 1; m >>= 1)
          for (int y = 1; y <= queries && y <= 64; ++y) {
            const int part = (queries + y - 1) / y;
            const long long ctas = (long long)((pl.n_tiles + m - 1) / m) * nh * ((queries + part - 1) / part);
            const double cost = (double)((ctas + 147) / 148) * (part * pl.n_mt * (m == 4 ? 4.0 : m == 2 ? 2.4 : 1.6) + 16.0);
            if (best == 0.0 || cost < best) {
              best = cost;
              per_cta = m;
              parts = part;
            }
          }
        rp.m_per_cta = per_cta;
        rp.tiles_per_split = parts * pl.n_mt;
        if (launch_pass(rel_pass_kernel<D, kMasses>, 2, pl.n_tiles, (queries + parts - 1) / parts * (kGroups / per_cta), nh) != ADAPSHOT_OK)
          return ADAPSHOT_ECUDA;
        rp.tiles_per_split = pl.tiles_per_split;
        ads_launch_dependent(rel_keys_kernel, dim3((unsigned)((pool->n_shots + 7) / 8), (unsigned)(b1 - b0 + 1)), 256, 0, st,
                             pieces, shot_off, pool->n_shots, nh, h0, (long long)pl.n_tiles * kTile, pool->pool_tokens, b0, mass);
        if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
        continue;
      }
      int warps = 8;                                                  // per shot: one where shots alone fill the chip
      while (warps > 1 && (long long)pool->n_shots * (b1 - b0 + 1) * warps > 2 * 8 * 148 * 4) warps >>= 1;
      ads_launch_dependent(rel_reduce_kernel, dim3((unsigned)((pool->n_shots + 8 / warps - 1) / (8 / warps)),
                           (unsigned)(b1 - b0 + 1)), 256, 0, st, pieces, ml_part, shot_off, pool->n_shots, nh, pl.n_mt, t0,
                           n, pl.splits, pl.tiles_per_split, pool->pool_tokens, b0, h0, warps, mass);
      if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    }

  const long long n_sc = (long long)B * pool->n_shots;
  ads_launch_dependent(rel_scores_kernel, (unsigned)((n_sc + 255) / 256), 256, 0, st, mass, shot_off, B, pool->n_shots, 1.0 / ((double)Tq * Hq),
      (flags & ADAPSHOT_RELEVANCE_PER_TOKEN) ? 1 : 0, keys);
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  return ads_topk_from_keys(keys, pool->n_shots, B, k, sel_idx, sel_score, st);
}

}  // namespace

extern "C" size_t adapshot_select_attn_workspace_bytes(const adapshot_model_t* model, const adapshot_pool_t* pool,
                                                       int32_t B, int32_t Tq, int32_t k) {
  if (model == nullptr || pool == nullptr || !rel_shape_ok(model) || B <= 0 || Tq <= 0 || k <= 0 ||
      pool->n_shots <= 0 || pool->pool_tokens <= 0)
    return 0;
  return rel_plan(model, pool, B, Tq).total;
}

extern "C" int adapshot_select_attn(const adapshot_model_t* model, const adapshot_pool_t* pool, int32_t layer,
                                    const void* q, int32_t B, int32_t Tq, int32_t k, uint32_t flags,
                                    int32_t* sel_idx, float* sel_score, void* ws, size_t ws_bytes,
                                    int32_t* status, void* stream) {
  if (model == nullptr || pool == nullptr || q == nullptr || sel_idx == nullptr || ws == nullptr)
    return ADAPSHOT_EINVAL;
  if (pool->k == nullptr || pool->shot_off == nullptr || pool->n_shots <= 0 || pool->pool_tokens <= 0 || B <= 0 ||
      Tq <= 0 || (flags & ~ADAPSHOT_RELEVANCE_PER_TOKEN) != 0)
    return ADAPSHOT_EINVAL;
  if (model->dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (!rel_shape_ok(model)) return ADAPSHOT_ESHAPE;
  if (layer < 0 || layer >= model->n_layers) return ADAPSHOT_ESHAPE;
  if (k < 1 || k > pool->n_shots) return ADAPSHOT_ESHAPE;
  if (pool->n_shots > 8192 && k > 4096) return ADAPSHOT_EUNSUPPORTED;
  if (pool->pool_tokens > (1ll << 31) - 256) return ADAPSHOT_ESHAPE;
  if (!ads_aligned16(pool->k) || !ads_aligned16(q) || ((uintptr_t)ws & 255u) || ((uintptr_t)pool->shot_off & 7u))
    return ADAPSHOT_EALIGN;
  const RelPlan pl = rel_plan(model, pool, B, Tq);
  if ((long long)B * pl.n_mt > 0x7fffffffll || pl.splits > 65535 || model->n_kv_heads > 65535) return ADAPSHOT_ESHAPE;
  if (ws_bytes < pl.total) return ADAPSHOT_ECAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (model->head_dim == 128)
    return rel_launch<128>(model, pool, layer, q, B, Tq, k, flags, sel_idx, sel_score, pl, ws, status, st);
  return rel_launch<64>(model, pool, layer, q, B, Tq, k, flags, sel_idx, sel_score, pl, ws, status, st);
}
