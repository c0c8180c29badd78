// Probe attention over the reused cache (paper Eq. 1 with the tree mask of Sec. 4.1:
// probe j sees the first n_j shots of the assembled context and, causally, its own
// tokens; scores scaled by 1/sqrt(d) as in Eq. 5; rotary positions of Eq. 6).
//
// Three kernels:
//   attn_prep     rotates Q and the probe's own K to their positions L_j + t, packs the
//                 Q rows of one KV head (GQA) into an M-major tile layout, and writes
//                 the schedule (how many 128-key tiles every (probe, query) pair has
//                 and where the tile sequence is cut into ranges of equal cost);
//   attn_main     persistent CTAs.  A CTA works on two 128-row M tiles of one KV head
//                 at a time ("M pair"): TMA stages each K/V tile once for both, one
//                 thread issues tcgen05 UMMAs (S = Q K^T, O += P V, accumulators in
//                 TMEM, P kept in TMEM), two groups of four warps run the online
//                 softmax of the two M tiles (one thread per row) and alternate on the
//                 tensor pipe.  The global tile sequence is cut into ranges of equal
//                 cost, one per gang of CTAs (the CTAs of a gang take the M pairs of the
//                 same K/V tiles, so the tiles are shared through L2).  A range that
//                 covers a whole unit stores the final bf16 rows (staged through shared
//                 memory into whole row segments); a range that cuts a unit stores
//                 un-normalised partials;
//   attn_combine  log-sum-exp merge of the partials of the cut units.
// Two variants take tiles straight from the pool, through a row map that the preparation writes once per call: the
// V-from-pool variant (adapshot_query_attn_vpool) reads K from a cache that holds the re-encoded K only and
// V, which Eq. 7 leaves as it is, from the pool, so that the gather moves half the bytes; the fused variant
// (adapshot_query_attn_fused) reads both from the pool and re-encodes K (Eq. 7) in shared memory.  One warp per
// operand stitches a tile from the runs of pool rows it consists of; four warps rotate K where it landed.
// (Fused, 2 queries x 2 layers x 16.4 K tokens, probes of 64 and 128 shots: 1396 us with two warps that copied K
// and V element-wise and rotated K from a table, 535 us with four warps that rotated K on its way through
// registers (16 KB in flight per SM, latency-bound), 325 us as it is now.)
#include <cuda.h>
#include <float.h>
#include <string.h>

#include "common.cuh"
#include "entropy.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.cuh"

namespace {

using namespace sm100;

constexpr int kMaxProbes = 16;
constexpr int kMaxPairs = 256;       // (probe, query) pairs one call may hold: B * P <= 256
constexpr int kMaxCtas = 160;        // persistent grid: one CTA per SM, at most this many
constexpr int kMaxGang = 8;          // CTAs that share one range of K/V tiles
// Fixed cost of starting a unit, in tiles.  (10 k clocks when every role walked the schedule by itself, 3 k of them the walk that one thread does
// ahead now.  2 / 3 / 4 / 6, us: one layer of one query, four probes 122.8 / 122.9 / 123.9 / 124.9, two rounds of probes 569 / 567 / 572 / 572, 28 queries
// of seven short probes 217 / 221 / 226 / 238, seven queries of four, eight layers 682 / 663 / 650 / 680: flat from 2 to 4.)
constexpr int kUnitCost = 4;
constexpr int kTileM = 128;          // query rows per M tile (TMEM lanes)
constexpr int kTileN = 128;          // keys per tile
constexpr int kAttnThreads = 384;    // warp 0 TMA and items, warp 1 MMA, warp 2 gathers V (V from the pool), softmax of M tile A on
                                     // warps 4-7, B on 8-11
constexpr int kFusedThreads = 512;   // fused variant: warps 2-3 gather V and K, softmax on warps 4-11, K rotated by warps 12-15
constexpr int kModeCache = 0;        // K and V tiles by TMA from the assembled cache
constexpr int kModeFused = 1;        // K and V tiles from the pool, K re-encoded in shared memory
constexpr int kModeVPool = 2;        // K tiles by TMA from a K-only cache, V tiles from the pool
constexpr int kRotateWarp0 = 12;     // fused variant: first of the four warps that rotate K
constexpr int kRotateWarps = 4;
// Registers per thread of the warpgroups (TMA / MMA / gather, softmax twice): together what 384 threads are launched
// with, 3 x 168.
constexpr int kRegsIssue = 120, kRegsSoftmax = 192;
static_assert(kRegsIssue + 2 * kRegsSoftmax <= 3 * 168, "register split");
// Registers per thread of the fused variant's warpgroups (issue and gather, softmax twice, rotation): together
// what 512 threads are launched with, 4 x 128.
constexpr int kFusedRegsIssue = 64, kFusedRegsSoftmax = 176, kFusedRegsRotate = 96;
static_assert(kFusedRegsIssue + 2 * kFusedRegsSoftmax + kFusedRegsRotate <= 4 * 128, "register split");
constexpr uint32_t kTmemCols = 512;
constexpr float kRescaleThreshold = 8.f;   // log2 units: rescale O only when the max grows by 2^8
constexpr float kNegSentinel = -1.0e30f;
constexpr float kLn2 = 0.6931471805599453f;

// Schedule shared by the main and the combine kernel (lives in the workspace).
// Pairs are ordered longest probe first: pair = (P-1-j) * B + b.  Every pair owns
// nl * Hkv units (layer, kv head) of n_su tiles each: n_ctx context tiles followed by
// n_own tiles of the probe's own tokens.  The ranges are equal in cost, not in tiles: every
// unit that starts in a range adds kUnitCost tiles' worth of time to it (Q load and pipeline
// fill, read-out of O), which matters when the units are as short as a range.
struct Sched {
  long long total;                   // tiles of all units
  long long start[kMaxCtas + 1];     // first tile of every gang's range; start[n_gangs] = total
  int first_pair[kMaxCtas + 1];      // pair that holds start[q]
  long long prefix[kMaxPairs + 1];   // first tile of every pair in the global sequence
  long long Lj[kMaxPairs];           // context length of the pair's probe (clamped to ctx_cap)
  int n_ctx[kMaxPairs];
  int n_su[kMaxPairs];
  int n_cut;                         // units that a range boundary cuts; their pieces are merged afterwards
  struct Cut {
    int bpj, g;                      // (b * nl + l) * P + j and KV head of the unit
    int gang, n;                     // its pieces lie with gangs gang .. gang + n - 1
    int which;                       // slot of the first piece (the others are their gangs' first pieces)
  } cut[kMaxCtas];
};

struct AttnParams {
  const Sched* sched;
  float* o_part;              // [slots][2][D/4][128][4] fp32, un-normalised (rows contiguous per 4 columns)
  float* ml_part;             // [slots][2][128][2]  (running max in log2 units, row sum)
  __nv_bfloat16* out;         // [B][nl][P][Tq][Hq][D]
  float* lse;                 // [B][nl][P][Hq][Tq] or null
  int32_t* status;
  int B, P, Tq, Hq, Hkv, G, nl;
  int To;                     // own tokens per probe (>= Tq): the Tq rows are the last Tq of them
  int n_mt, n_mp, gang, n_gangs;
  float scale_log2;           // softmax_scale * log2(e)
  unsigned long long g_magic; // ceil(2^32 / G)
  // K or V from the pool
  const int* row_map;            // [B][ctx_cap]: pool token of every context position, -1 beyond L
  const int* off_map;            // [B][ctx_cap]: first position of the shot a position lies in (k_pos_mode 1)
  int k_pos_mode;                // 0: angle = position; 1: angle = the shot's first position (Eq. 7 as printed)
  long long ctx_cap;
  int layer_begin;
  double theta[64];
};

// V-from-pool and fused variants, once per call: the pool token behind every context position of every query
// (the gather's plan lookup, stored instead of applied) and, for keys stored rotated, the first position of its
// shot.  Positions from L to the end of the last 128-token tile get -1; nothing beyond them is read.
struct RowMapParams {
  const long long* ctx_off;   // [B][k+1]
  const int32_t* sel_idx;     // [B][k]
  const long long* shot_off;  // [n_shots+1]
  int* row_map;               // [B][ctx_cap]
  int* off_map;               // [B][ctx_cap] or null
  long long ctx_cap;
  int B, k, n_shots;
};

struct PrepParams {
  const __nv_bfloat16* q;     // [B][nl][P][Tq][Hq][D]
  const __nv_bfloat16* kq;    // [B][nl][P][To][Hkv][D]
  __nv_bfloat16* q_rot;       // [B*nl*P*Hkv][Tq*G][D]
  __nv_bfloat16* kq_rot;      // layout of kq
  const long long* ctx_off;
  Sched* sched;
  long long ctx_cap;
  int B, k, P, Tq, Hq, Hkv, nl, n_gangs;
  int To;                     // own tokens per probe: the Tq query rows are the last Tq of them
  const int* nshots_dev;      // per-query shot count of the (single) probe, device memory, or null
  int32_t* status;
  double theta[64];           // theta_i = rope_base^(-2i/D), formed on the host
  int nshots[kMaxProbes];
  // what else the launch does: its blocks are the schedule's, then these, then the tokens'
  AdsEntropyJob ent;          // entropy of the probes' logits, first step
  RowMapParams map;
  int map_blocks;             // eight selected shots each; 0: no row map
  int tok_blocks;
};

__device__ __forceinline__ void bf16x8_unpack(const uint4& r, float* x) {
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    x[2 * j] = __uint_as_float(w[j] << 16);
    x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
  }
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint4 bf16x8_pack(const float* x) {
  return make_uint4(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]), pack_bf16x2(x[4], x[5]),
                    pack_bf16x2(x[6], x[7]));
}

constexpr int kPrepParts = 4;

// Shots of probe j of query b: from the host list, or (decode over the prefix each query chose)
// from a per-query device array; a count outside 1..k is reported and clamped.
__device__ __forceinline__ int probe_shots(const PrepParams& p, int b, int j) {
  if (p.nshots_dev == nullptr) return p.nshots[j];
  int n = p.nshots_dev[b];
  if (n < 1 || n > p.k) {
    ads_set_status(p.status, ADAPSHOT_EINDEX);
    n = n < 1 ? 1 : p.k;
  }
  return n;
}

// One warp (w) per selected shot: its run of positions is written with whole lines (a search per position
// took 38 us for 32 queries of 66 K positions and 8.3 us for 8 of 33 K; 3 us for those now).
__device__ __forceinline__ void row_map_warp(const RowMapParams& p, long long w, int lane) {
  if (w >= (long long)p.B * p.k) return;
  const int b = (int)(w / p.k), r = (int)(w % p.k);
  const long long* off = p.ctx_off + (long long)b * (p.k + 1);
  const long long o0 = off[r], o1 = off[r + 1];
  const int s = p.sel_idx[w];
  int* rows = p.row_map + (long long)b * p.ctx_cap;
  int* firsts = p.off_map == nullptr ? nullptr : p.off_map + (long long)b * p.ctx_cap;
  const long long end = min(o1, p.ctx_cap);
  const bool known = s >= 0 && s < p.n_shots;        // (an unknown shot is reported by the plan and has no positions)
  const long long src = known ? p.shot_off[s] - o0 : 0;
  for (long long pos = o0 + lane; pos < end; pos += 32) {
    rows[pos] = known ? (int)(src + pos) : -1;
    if (firsts != nullptr) firsts[pos] = (int)o0;
  }
  if (r == p.k - 1) {
    const long long pad = min((o1 + kTileN - 1) / kTileN * kTileN, p.ctx_cap);
    for (long long pos = o1 + lane; pos < pad; pos += 32) {
      rows[pos] = -1;
      if (firsts != nullptr) firsts[pos] = 0;
    }
  }
}

// kPrepParts warps per own token (b, l, j, u): all Hq query heads and Hkv key heads of the token rotate by the same
// angles (L_j + u) * theta_i, which the block forms once for its tokens, half an angle per thread, while the first
// rows are on their way.  (Every lane forming its eight angles itself was what bound the kernel: 4096 tokens of 32
// + 8 heads, 84 MB, 27 us and 14336 tokens 82-90 us; 20 and 73 then.)  The blocks stay for the whole call: the angles of their next
// tokens, a chain of two loads and fp64 arithmetic, are formed while this group's rows are on their way (a block per two tokens: 21.2 and
// 73 us, 17.2 and 60 now).  The first block writes the schedule instead: started
// first, its chain of dependent steps lies under the others' copies.
template <int D>
__global__ void __launch_bounds__(256, 3) attn_prep_kernel(const __grid_constant__ PrepParams p) {
  constexpr int VPH = D / 8, HALF_V = VPH / 2;
  const int lane = threadIdx.x & 31;
  ads_dependency_wait();

  if (blockIdx.x == 0) {
    // the schedule, by a block of its own (beside the rotation, not in front of a share of it);
    // intermediate values stay in shared memory.  One pair per thread (kMaxPairs = blockDim.x): the
    // prefix sums are a block scan.
    __shared__ long long s_pre[kMaxPairs + 1], s_vpre[kMaxPairs + 1], s_start[kMaxCtas + 1], s_warp[2][8];
    __shared__ int s_nsu[kMaxPairs], s_fp[kMaxCtas + 1], s_ncut;
    Sched* sc = p.sched;
    const int n_pairs = p.P * p.B, pi = threadIdx.x;
    const int n_own = (p.To + kTileN - 1) / kTileN;
    const long long units_per_pair = (long long)p.nl * p.Hkv;
    long long len = 0, vlen = 0;
    if (pi < n_pairs) {
      const int j = p.P - 1 - pi / p.B, b = pi % p.B;
      long long Lj = p.ctx_off[(long long)b * (p.k + 1) + probe_shots(p, b, j)];
      Lj = Lj > p.ctx_cap ? p.ctx_cap : (Lj < 0 ? 0 : Lj);
      const int n_ctx = (int)((Lj + kTileN - 1) / kTileN);
      sc->Lj[pi] = Lj;
      sc->n_ctx[pi] = n_ctx;
      sc->n_su[pi] = n_ctx + n_own;
      s_nsu[pi] = n_ctx + n_own;
      len = (n_ctx + n_own) * units_per_pair;
      vlen = (n_ctx + n_own + kUnitCost) * units_per_pair;
    }
    if (pi == 0) s_ncut = 0;
    long long in_l = len, in_v = vlen;                // inclusive scans
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long a = __shfl_up_sync(0xffffffffu, in_l, o), c = __shfl_up_sync(0xffffffffu, in_v, o);
      if (lane >= o) { in_l += a; in_v += c; }
    }
    if (lane == 31) { s_warp[0][pi >> 5] = in_l; s_warp[1][pi >> 5] = in_v; }
    __syncthreads();
    for (int w = 0; w < (pi >> 5); ++w) { in_l += s_warp[0][w]; in_v += s_warp[1][w]; }
    if (pi < n_pairs) {
      s_pre[pi] = in_l - len;
      s_vpre[pi] = in_v - vlen;
      sc->prefix[pi] = in_l - len;
      if (pi == n_pairs - 1) {
        s_pre[n_pairs] = in_l;
        s_vpre[n_pairs] = in_v;
        sc->prefix[n_pairs] = in_l;
        sc->total = in_l;
      }
    }
    __syncthreads();
    // Range q starts where the cost sequence (every unit preceded by kUnitCost virtual tiles)
    // reaches q / n_ranges of its length: threads q = 0 .. n_gangs, independently.  A range is at least
    // kUnitCost + 1 long, so that it holds a real tile: a call with less work leaves gangs without any.
    const long long vtotal = s_vpre[n_pairs];
    const long long fit = vtotal / (kUnitCost + 1);
    const int n_ranges = (int)(fit < 1 ? 1 : (fit < p.n_gangs ? fit : p.n_gangs));
    for (int q = threadIdx.x; q <= p.n_gangs; q += blockDim.x) {
      const long long v = q < n_ranges ? q * vtotal / n_ranges : vtotal;
      long long real = s_pre[n_pairs];
      int fp = n_pairs - 1;
      if (v < vtotal) {
        int lo = 0, hi = n_pairs;                   // pair with s_vpre[lo] <= v < s_vpre[lo + 1]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (s_vpre[mid] <= v) lo = mid; else hi = mid;
        }
        const long long lv = s_nsu[lo] + kUnitCost;
        const long long rel = v - s_vpre[lo];
        const long long su = rel / lv, off = rel % lv;
        real = s_pre[lo] + su * s_nsu[lo] + (off > kUnitCost ? off - kUnitCost : 0);
        fp = lo;
      }
      sc->start[q] = real;
      sc->first_pair[q] = fp;
      s_start[q] = real;
      s_fp[q] = fp;
    }
    __syncthreads();
    // The units to merge: gang q lists the unit that its range's end cuts, if the unit starts in that range.
    for (int q = threadIdx.x; q + 1 < n_ranges; q += blockDim.x) {
      const long long cut = s_start[q + 1];
      const int pr = s_fp[q + 1];
      const long long nsu = s_nsu[pr], rel = cut - s_pre[pr];
      const long long su = rel / nsu, s_u = s_pre[pr] + su * nsu;
      if (s_u == cut || s_u < s_start[q]) continue;   // between two units; or an earlier gang holds its first piece
      int n = 2;                                      // gangs whose range begins inside the unit, and this one
      while (q + n < n_ranges && s_start[q + n] < s_u + nsu) ++n;
      Sched::Cut c;
      const int l = (int)(su / p.Hkv);
      c.bpj = ((pr % p.B) * p.nl + l) * p.P + p.P - 1 - pr / p.B;
      c.g = (int)(su % p.Hkv);
      c.gang = q;
      c.n = n;
      c.which = s_start[q] >= s_u ? 0 : 1;
      sc->cut[atomicAdd(&s_ncut, 1)] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) sc->n_cut = s_ncut;
    return;
  }
  int blk = (int)blockIdx.x - 1;
  if (blk < p.ent.blocks) {
    if (p.ent.f32)
      ent_partial_block(static_cast<const float*>(p.ent.logits), p.ent.V, p.ent.row_stride, p.ent.slice, p.ent.n_split, p.ent.partial, blk);
    else
      ent_partial_block(static_cast<const __nv_bfloat16*>(p.ent.logits), p.ent.V, p.ent.row_stride, p.ent.slice, p.ent.n_split,
                        p.ent.partial, blk);
    return;
  }
  blk -= p.ent.blocks;
  if (blk < p.map_blocks) {
    row_map_warp(p.map, blk * 8ll + (threadIdx.x >> 5), lane);
    return;
  }
  blk -= p.map_blocks;
  constexpr int kTokens = 8 / kPrepParts;           // of a block at a time
  __shared__ float2 angle_s[2][kTokens][D / 2];     // (cos, sin)
  // (tokens and rows fit 32 bits: 2^31 of them would not fit the device's memory)
  const int n_tok = p.B * p.nl * p.P * p.To, n_groups = (n_tok + kTokens - 1) / kTokens;
  const int warp = threadIdx.x >> 5, slot = warp / kPrepParts, part = warp % kPrepParts;
  const int G = p.Hq / p.Hkv, jcol = lane % HALF_V;
  constexpr int kFly = 3;                           // units of a lane loaded at once (the 8B shape has 2.5 per lane)
  uint4 lo[kFly], hi[kFly];
  int tok, bpj, t, units;                           // of this thread's token
  auto take = [&](int group) {
    tok = group * kTokens + slot;
    bpj = tok / p.To;                               // (b*nl + l)*P + j
    t = tok - bpj * p.To - (p.To - p.Tq);           // query row of this token (the last Tq own tokens have one), or negative
    units = tok < n_tok ? (p.Hq + p.Hkv) * HALF_V : 0;
  };
  auto load = [&](int u0) {
    const uint4* qsrc = reinterpret_cast<const uint4*>(p.q) + ((long long)bpj * p.Tq + max(t, 0)) * p.Hq * VPH + jcol;
    const uint4* ksrc = reinterpret_cast<const uint4*>(p.kq) + (long long)tok * p.Hkv * VPH + jcol;
#pragma unroll
    for (int e = 0; e < kFly; ++e) {
      const int u = u0 + e * 32 * kPrepParts, head = u / HALF_V;       // column == jcol since 32 % HALF_V == 0
      if (u >= units || (head < p.Hq && t < 0)) continue;
      const uint4* src = head < p.Hq ? qsrc + head * VPH : ksrc + (head - p.Hq) * VPH;
      lo[e] = src[0];
      hi[e] = src[HALF_V];
    }
  };
  auto angles = [&](int group, int buf) {
    for (int i = threadIdx.x; i < kTokens * (D / 2); i += 256) {
      const int tk = group * kTokens + i / (D / 2);
      if (tk < n_tok) {
        const int x = tk / p.To, bl = x / p.P, j = x - bl * p.P, b = bl / p.nl;
        const long long Lj = p.ctx_off[(long long)b * (p.k + 1) + probe_shots(p, b, j)];
        float sn, cs;
        rope_sincos((double)(Lj + tk - x * p.To), p.theta[i % (D / 2)], &sn, &cs);
        angle_s[buf][i / (D / 2)][i % (D / 2)] = make_float2(cs, sn);
      }
    }
  };
  const int u_first = part * 32 + lane;
  take(blk);
  load(u_first);
  angles(blk, 0);
  __syncthreads();
  for (int group = blk, buf = 0; group < n_groups; group += p.tok_blocks, buf ^= 1) {
    const int next = group + p.tok_blocks;
    if (next < n_groups) angles(next, buf ^ 1);      // (under the loads of this group's rows)
    float sn[8], cs[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 v = *reinterpret_cast<const float4*>(&angle_s[buf][slot][jcol * 8 + 2 * e]);
      cs[2 * e] = v.x; sn[2 * e] = v.y; cs[2 * e + 1] = v.z; sn[2 * e + 1] = v.w;
    }
    for (int u0 = u_first; u0 < units; u0 += kFly * 32 * kPrepParts) {
      if (u0 >= kFly * 32 * kPrepParts) load(u0);
#pragma unroll
      for (int e = 0; e < kFly; ++e) {
        const int u = u0 + e * 32 * kPrepParts, head = u / HALF_V;
        if (u >= units || (head < p.Hq && t < 0)) continue;
        float x[8], y[8], xr[8], yr[8];
        bf16x8_unpack(lo[e], x);
        bf16x8_unpack(hi[e], y);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          xr[c] = x[c] * cs[c] - y[c] * sn[c];
          yr[c] = y[c] * cs[c] + x[c] * sn[c];
        }
        uint4* dst;
        if (head < p.Hq) {
          const int g = head / G, hh = head - g * G;
          const long long row = ((long long)bpj * p.Hkv + g) * (p.Tq * G) + t * G + hh;
          dst = reinterpret_cast<uint4*>(p.q_rot) + row * VPH + jcol;
        } else {
          dst = reinterpret_cast<uint4*>(p.kq_rot) + (long long)tok * p.Hkv * VPH + (head - p.Hq) * VPH + jcol;
        }
        dst[0] = bf16x8_pack(xr);
        dst[HALF_V] = bf16x8_pack(yr);
      }
    }
    if (next < n_groups) {
      take(next);
      load(u_first);
    }
    __syncthreads();
  }
}

// Shared-memory plan.  Every operand tile is made of [128 rows][128 bytes] sub-tiles
// written by TMA with the 128-byte swizzle; D = 128 needs two of them per tile.
// The fused variant has a third K stage (one tile landing, one being rotated, one in use) in the place of
// the read-out staging.
constexpr int kCachePairs = 12;       // (30 of them: no faster, 192 short pairs in one range 2234.5 / 2234.7 us)
constexpr uint32_t kCacheBytes = 320;
constexpr uint32_t kBarBytes = 384;                  // barriers, TMEM slot, abort flags
constexpr int kItems = 4;                            // items published ahead of the roles that work on them
template <int D, int MODE>
struct AttnSmem {
  static constexpr int kKStages = MODE == kModeFused ? 3 : 2;
  static constexpr int kVStages = 2;
  static constexpr uint32_t kStageBytes = MODE == kModeFused ? 0 : 4096;  // per softmax warp: 32 rows x 128 bytes
  static constexpr uint32_t kTileBytes = (D / 64) * 16384u;
  static constexpr uint32_t kOffQ = 0;                                    // Q of M tile A, then of M tile B
  static constexpr uint32_t kOffK = kOffQ + 2 * kTileBytes;
  static constexpr uint32_t kOffV = kOffK + kKStages * kTileBytes;
  static constexpr uint32_t kOffStage = kOffV + kVStages * kTileBytes;    // read-out staging of the 8 softmax warps
  static constexpr uint32_t kOffBar = kOffStage + 8 * kStageBytes;
  static constexpr uint32_t kOffItems = kOffBar + kBarBytes;
  static constexpr uint32_t kOffCache = kOffItems + kItems * 64;
  static constexpr uint32_t kOffRows = kOffCache + kCacheBytes;                   // pool rows of a tile, per gather warp
  static constexpr uint32_t kTotal = kOffRows + (MODE == kModeVPool ? 512 : MODE == kModeFused ? 1024 : 0) + 1024;   // + alignment slack
};

// mbarrier slots (8 bytes each)
enum Bar {
  kBarQFull = 0, kBarQEmpty = 2, kBarKFull = 4, kBarKEmpty = 7, kBarVFull = 10, kBarVEmpty = 13,
  kBarSFull = 16, kBarPFull = 18, kBarOFull = 20, kBarOEmpty = 22, kBarDrain = 24,
  kBarKRot = 25,                 // fused variant: K tile rotated
  kBarItemFull = 28, kBarItemEmpty = 28 + kItems,
  kNumBars = 28 + 2 * kItems
};
static_assert(8 * kNumBars + 16 <= kBarBytes, "room of the barriers");

// A piece = the part of one unit (pair, layer, kv head) that falls into a gang's range.
struct Piece {
  int pair, su, t0, t1, n_su, n_ctx;
  long long Lj;
  bool first_of_gang;
};

struct Walker {
  long long x, begin, end;
  int pair;                      // pair that holds x (pieces only move forward)
};

// The part of the schedule a CTA walks, copied to shared memory once: the pairs from the
// one its range starts in.  Pairs beyond the copy (a range that spans more than
// kCachePairs pairs) are read from the workspace.
struct SchedCache {
  long long prefix[kCachePairs + 1];
  long long Lj[kCachePairs];
  int n_ctx[kCachePairs];
  int n_su[kCachePairs];
  long long begin, end;
  int p0, n;
};
static_assert(sizeof(SchedCache) <= kCacheBytes, "room of the schedule cache");
struct PairInfo {
  long long prefix, next_prefix, Lj;
  int n_ctx, n_su;
};
__device__ __forceinline__ PairInfo pair_info(const Sched* sc, const SchedCache* c, int pair) {
  PairInfo pi;
  const int k = pair - c->p0;
  if (k >= 0 && k < c->n) {
    pi.prefix = c->prefix[k]; pi.next_prefix = c->prefix[k + 1]; pi.Lj = c->Lj[k];
    pi.n_ctx = c->n_ctx[k]; pi.n_su = c->n_su[k];
  } else {
    pi.prefix = sc->prefix[pair]; pi.next_prefix = sc->prefix[pair + 1]; pi.Lj = sc->Lj[pair];
    pi.n_ctx = sc->n_ctx[pair]; pi.n_su = sc->n_su[pair];
  }
  return pi;
}

__device__ __forceinline__ bool next_piece(const Sched* sc, const SchedCache* cache, int n_pairs, Walker& wk,
                                           Piece& pc) {
  if (wk.x >= wk.end) return false;
  PairInfo pi = pair_info(sc, cache, wk.pair);
  while (wk.pair + 1 < n_pairs && pi.next_prefix <= wk.x) pi = pair_info(sc, cache, ++wk.pair);
  const int lo = wk.pair;
  const int nsu = pi.n_su;
  const long long rel = wk.x - pi.prefix;
  pc.pair = lo;
  // (a 32-bit division where the position allows it: the 64-bit one is some hundred dependent instructions)
  pc.su = (rel >> 32) == 0 ? (int)((uint32_t)rel / (uint32_t)nsu) : (int)(rel / nsu);
  pc.t0 = (int)(rel - (long long)pc.su * nsu);
  const long long room = wk.end - wk.x;
  pc.t1 = (int)(room < (long long)(nsu - pc.t0) ? pc.t0 + room : nsu);
  pc.n_su = nsu;
  pc.n_ctx = pi.n_ctx;
  pc.Lj = pi.Lj;
  pc.first_of_gang = wk.x == wk.begin;
  wk.x += pc.t1 - pc.t0;
  return true;
}

// One M pair of one piece: what a CTA works on between two read-outs of O.  One thread walks the schedule and publishes the
// items in shared memory, a few ahead: each of ten roles walking it by itself paid 3000 clocks of dependent divisions between
// two items, and the issuing thread's and the softmax warps' were in the chain (four probes of 4 to 16 shots, 16 layers: 603 -> 582 us
// with the rounds' other kernels, no cache 343 -> 308; seven probes of 32 queries 6240 -> 6150).
struct __align__(64) Item {
  int n_tiles;                   // -1: no more items
  int n_ctx, ctx_begin, own_begin;
  int b, l, g, mp;
  int flags;                     // 1: there is an M tile B; 2: the piece covers its unit
  int outer_ctx, outer_own, outer_q;
  int Lj, slot;
  __device__ bool has_b() const { return (flags & 1) != 0; }
  __device__ bool whole() const { return (flags & 2) != 0; }
};
static_assert(sizeof(Item) == 64, "room of an item");

__device__ __forceinline__ void make_item(const AttnParams& p, const Piece& pc, int gang_id, int mp, Item& w) {
  const int j = p.P - 1 - pc.pair / p.B;
  w.b = pc.pair % p.B;
  w.l = pc.su / p.Hkv;
  w.g = pc.su - w.l * p.Hkv;
  w.mp = mp;
  w.flags = (2 * mp + 1 < p.n_mt ? 1 : 0) | (pc.t0 == 0 && pc.t1 == pc.n_su ? 2 : 0);
  w.Lj = (int)pc.Lj;
  const int ctx_end = min(pc.t1, pc.n_ctx);
  w.ctx_begin = pc.t0;
  w.n_ctx = max(0, ctx_end - pc.t0);
  // own-token tiles this M pair can see (causal): tokens up to the pair's last row
  const int row_hi = min(p.Tq * p.G - 1, mp * 2 * kTileM + 2 * kTileM - 1);
  const int own_need = (p.To - p.Tq + row_hi / p.G) / kTileN + 1;
  w.own_begin = max(pc.t0, pc.n_ctx) - pc.n_ctx;
  const int own_end = min(pc.t1 - pc.n_ctx, own_need);
  const int n_own = max(0, own_end - w.own_begin);
  w.n_tiles = w.n_ctx + n_own;
  w.outer_ctx = w.b * p.nl + w.l;
  w.outer_own = w.outer_ctx * p.P + j;
  w.outer_q = w.outer_own * p.Hkv + w.g;
  w.slot = (2 * gang_id + (pc.first_of_gang ? 0 : 1)) * p.n_mp + mp;
}

// m / G for 0 <= m < 2^32 with g_magic = ceil(2^32 / G)
__device__ __forceinline__ int div_g(const AttnParams& p, int m) {
  uint32_t q = (uint32_t)(((unsigned long long)(uint32_t)m * p.g_magic) >> 32);     // at most one too large
  if (q * (uint32_t)p.G > (uint32_t)m) --q;
  return (int)q;
}

// Maps over the pool's V (or K) with boxes of 1, 2, 4, ..., 128 rows, from which a tile is stitched run by
// run (a run = consecutive context positions that are consecutive pool rows).
struct PoolMaps {
  CUtensorMap m[8];
};

// TMEM: S/P of M tile A at columns 0..127, of M tile B at 128..255 (P, as packed bf16,
// overwrites the S tile it was computed from); O accumulators at 256 and 384.
// VPOOL and FUSED: V tiles are stitched from the pool by a gather warp.  FUSED: so are the K tiles, by a second
// one; four warps then re-encode them (Eq. 7) where they lie, so that no re-encoded cache is ever written to HBM.
template <int D, int MODE>
__global__ void __launch_bounds__(MODE == kModeFused ? kFusedThreads : kAttnThreads, 1)
attn_main_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kctx,
                 const __grid_constant__ CUtensorMap tm_vctx, const __grid_constant__ CUtensorMap tm_kown,
                 const __grid_constant__ CUtensorMap tm_vown, const __grid_constant__ PoolMaps vmaps,
                 const __grid_constant__ PoolMaps kmaps, const __grid_constant__ AttnParams p) {
  constexpr bool FUSED = MODE == kModeFused;
  constexpr bool VPOOL = MODE == kModeVPool;
  using SM = AttnSmem<D, MODE>;
  constexpr int SUB = D / 64;
  constexpr int KS = SM::kKStages, VS = SM::kVStages;
  constexpr uint32_t kTileBytes = SM::kTileBytes;
  constexpr uint32_t kIdescQK = idesc_bf16_f32(kTileM, kTileN, 0);
  constexpr uint32_t kIdescPV = idesc_bf16_f32(kTileM, D, 1);
  constexpr uint32_t kTmemS = 0, kTmemO = 256;
  constexpr int kSoftmaxWarp0 = 4;          // first of the eight softmax warps
  constexpr int kGatherWarp = 2;   // the warp that gathers the V tiles (fused: K by the next one)
  constexpr int kItemReaders = 8 + (FUSED ? 3 + kRotateWarps : VPOOL ? 2 : 1);     // every role's warps but the TMA thread's
  constexpr int kBarKReady = FUSED ? kBarKRot : kBarKFull;

  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_raw + (base - raw_addr);
  const uint32_t bar0 = base + SM::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * i; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + SM::kOffBar + 8 * kNumBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + SM::kOffBar + 8 * kNumBars + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_pairs = p.P * p.B;
  const int gang_id = blockIdx.x / p.gang, rank = blockIdx.x % p.gang;
  const Sched* sc = p.sched;

  if (threadIdx.x == 32) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(kBarQFull + i), 1);
      mbar_init(bar(kBarQEmpty + i), 1);
      mbar_init(bar(kBarSFull + i), 1);
      mbar_init(bar(kBarPFull + i), 4);
      mbar_init(bar(kBarOFull + i), 1);
      mbar_init(bar(kBarOEmpty + i), 4);
    }
    mbar_init(bar(kBarDrain), 1);
    for (int i = 0; i < 3; ++i) {
      mbar_init(bar(kBarKFull + i), 1);
      mbar_init(bar(kBarKEmpty + i), 1);
      mbar_init(bar(kBarVFull + i), 1);
      mbar_init(bar(kBarKRot + i), kRotateWarps);
      mbar_init(bar(kBarVEmpty + i), 1);
    }
    for (int i = 0; i < kItems; ++i) {
      mbar_init(bar(kBarItemFull + i), 1);
      mbar_init(bar(kBarItemEmpty + i), kItemReaders);
    }
    abort_flag[0] = 0;
    abort_flag[1] = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
    tmem_relinquish();
  } else if (warp == 3) {                    // the maps the mode uses: parameters of the kernel, so ahead of the wait
    if (lane == 0) tma_prefetch_desc(&tm_q);
    if (lane == 1) tma_prefetch_desc(&tm_kown);
    if (lane == 2) tma_prefetch_desc(&tm_vown);
    if (lane == 3 && !FUSED) tma_prefetch_desc(&tm_kctx);
    if (lane == 4 && MODE == kModeCache) tma_prefetch_desc(&tm_vctx);
    if (lane >= 8 && lane < 16 && MODE != kModeCache) tma_prefetch_desc(&vmaps.m[lane - 8]);
    if (lane >= 16 && lane < 24 && FUSED) tma_prefetch_desc(&kmaps.m[lane - 16]);
  }
  ads_dependency_wait();
  // the CTA's part of the schedule, fetched by two warps while the rest is set up
  SchedCache* cache = reinterpret_cast<SchedCache*>(base_ptr + SM::kOffCache);
  if (warp >= 2 && warp < 4) {
    const int p0 = sc->first_pair[gang_id];
    const int n = min(kCachePairs, n_pairs - p0);
    for (int k = threadIdx.x - 64; k <= n; k += 64) {
      cache->prefix[k] = sc->prefix[p0 + k];
      if (k < n) {
        cache->Lj[k] = sc->Lj[p0 + k];
        cache->n_ctx[k] = sc->n_ctx[p0 + k];
        cache->n_su[k] = sc->n_su[p0 + k];
      }
    }
    if (threadIdx.x == 64) {
      cache->begin = sc->start[gang_id];
      cache->end = sc->start[gang_id + 1];
      cache->p0 = p0;
      cache->n = n;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // ---- items: published by the TMA thread, read by a warp (or one thread of it) at a time
  Item* items = reinterpret_cast<Item*>(base_ptr + SM::kOffItems);
  // The n-th item; false at the end, or when the wait was given up (ok).  whole_warp: every lane calls and gets the item.
  auto read_item = [&](uint32_t n, Item& w, bool& ok, bool whole_warp) -> bool {
    const uint32_t slot = n % kItems;
    ok = mbar_wait(bar(kBarItemFull + slot), (n / kItems) & 1, abort_flag);
    if (whole_warp) ok = __all_sync(0xffffffffu, ok);
    if (!ok) return false;
    w = items[slot];
    if (whole_warp) __syncwarp();
    if (!whole_warp || lane == 0) mbar_arrive(bar(kBarItemEmpty + slot));
    return w.n_tiles >= 0;
  };

  auto role_tma = [&]() {
    // ------------------------------------------- TMA producer, and the walk through the schedule
    if (lane == 0) {
      Walker wk;
      wk.x = wk.begin = cache->begin;
      wk.end = cache->end;
      wk.pair = cache->p0;
      Piece pc;
      int mp = p.n_mp;                     // M pair of the next item; n_mp: the next piece's first
      uint32_t n_pub = 0;
      auto publish = [&](Item& w) -> bool {
        const uint32_t slot = n_pub % kItems;
        w.n_tiles = -1;
        if (mp >= p.n_mp && next_piece(sc, cache, n_pairs, wk, pc)) mp = rank;
        if (mp < p.n_mp) {
          make_item(p, pc, gang_id, mp, w);
          mp += p.gang;
        }
        if (!mbar_wait(bar(kBarItemEmpty + slot), ((n_pub / kItems) & 1) ^ 1, abort_flag)) return false;
        items[slot] = w;
        mbar_arrive(bar(kBarItemFull + slot));
        ++n_pub;
        return true;
      };
      uint32_t tk = 0, tv = 0, nq[2] = {0, 0};
      Item w, next;
      bool ok = publish(w);
      while (ok && w.n_tiles >= 0) {
        for (int x = 0; x < (w.has_b() ? 2 : 1) && ok && w.n_tiles > 0; ++x) {
          ok = mbar_wait(bar(kBarQEmpty + x), (nq[x] & 1) ^ 1, abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar(kBarQFull + x), kTileBytes);
#pragma unroll
          for (int s = 0; s < SUB; ++s)
            tma_load_3d(base + SM::kOffQ + x * kTileBytes + s * 16384u, &tm_q, bar(kBarQFull + x), s * 64,
                        (2 * w.mp + x) * kTileM, w.outer_q);
          ++nq[x];
        }
        // the next item is worked out while the first tiles of this one are on their way
        const int n_load = FUSED ? 0 : w.n_tiles;
        if (ok && n_load == 0) ok = publish(next);
        for (int i = 0; i < n_load && ok; ++i) {
          const bool own = i >= w.n_ctx;
          const CUtensorMap* mk = own ? &tm_kown : &tm_kctx;
          const CUtensorMap* mv = own ? &tm_vown : &tm_vctx;
          const int row = own ? (w.own_begin + i - w.n_ctx) * kTileN : (w.ctx_begin + i) * kTileN;
          const int outer = own ? w.outer_own : w.outer_ctx;
          const int sk = tk % KS;
          ok = mbar_wait(bar(kBarKEmpty + sk), ((tk / KS) & 1) ^ 1, abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar(kBarKFull + sk), kTileBytes);
#pragma unroll
          for (int s = 0; s < SUB; ++s)
            tma_load_4d(base + SM::kOffK + sk * kTileBytes + s * 16384u, mk, bar(kBarKFull + sk), s * 64, w.g, row,
                        outer);
          ++tk;
          if constexpr (!VPOOL) {
            const int sv = tv % VS;
            ok = mbar_wait(bar(kBarVEmpty + sv), ((tv / VS) & 1) ^ 1, abort_flag);
            if (!ok) break;
            mbar_arrive_expect_tx(bar(kBarVFull + sv), kTileBytes);
#pragma unroll
            for (int s = 0; s < SUB; ++s)
              tma_load_4d(base + SM::kOffV + sv * kTileBytes + s * 16384u, mv, bar(kBarVFull + sv), s * 64, w.g,
                          row, outer);
            ++tv;
          }
          if (i == min(1, n_load - 1)) ok = publish(next);
        }
        w = next;
      }
      if (!ok && !FUSED) {
        // gave up: let the copies already in flight land before the CTA retires
        for (uint32_t t = tk > (uint32_t)KS ? tk - KS : 0; t < tk; ++t)
          mbar_wait(bar(kBarKFull + t % KS), (t / KS) & 1, abort_flag + 1);
        if constexpr (!VPOOL)
          for (uint32_t t = tv > (uint32_t)VS ? tv - VS : 0; t < tv; ++t)
            mbar_wait(bar(kBarVFull + t % VS), (t / VS) & 1, abort_flag + 1);
      }
      if (!ok) {
        for (int x = 0; x < 2; ++x)
          if (nq[x] > 0) mbar_wait(bar(kBarQFull + x), (nq[x] - 1) & 1, abort_flag + 1);
      }
    }
    __syncwarp();
  };
  // Descriptors as a constant high half plus a low half = (address >> 4) with an immediate per k-step.
  constexpr uint32_t kHi = smem_desc_hi_sw128(1024);
  const uint32_t q_lo0 = smem_desc_lo(base + SM::kOffQ, 16);
  const uint32_t k_lo0 = smem_desc_lo(base + SM::kOffK, 16);
  const uint32_t v_lo0 = smem_desc_lo(base + SM::kOffV, 16384);
  auto qk_step = [&](const int x, uint32_t k_lo, int ks) {
    const uint32_t o = ((ks / 4) * 16384u + (ks % 4) * 32u) >> 4;
    umma_ss_lohi(tmem_base + kTmemS + x * kTileN, q_lo0 + x * (kTileBytes >> 4) + o, kHi, k_lo + o, kHi, kIdescQK,
                 ks > 0 ? 1u : 0u);
  };
  auto issue_pv = [&](const int x, uint32_t v_stage, bool first) {
    const uint32_t v_lo = v_lo0 + v_stage * (kTileBytes >> 4);
    const uint32_t d = tmem_base + kTmemO + x * 128;
    const uint32_t a = tmem_base + kTmemS + x * kTileN;
    // A = P from TMEM: 16 bf16 keys of one k-step occupy 8 packed columns
    umma_ts_lohi(d, a, v_lo, kHi, kIdescPV, first ? 0u : 1u);
#pragma unroll
    for (int ks = 1; ks < kTileN / 16; ++ks)
      umma_ts_lohi(d, a + ks * 8, v_lo + ((ks * 2048u) >> 4), kHi, kIdescPV, 1u);
  };
  auto role_mma = [&]() {
    // -------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      // The tensor pipe takes only a few UMMAs ahead of the one it runs: whatever this thread does between two issues is
      // time the pipe may idle, so the per-tile path is kept short.  (A thread per M tile that takes turns with the other,
      // so that each waits and commits under the other's UMMAs, is slower: one layer of one query 119.9 -> 126.9 us, eight
      // queries of 33 K tokens, four layers, 2765 -> 2880.)
      uint32_t tk = 0, tv = 0, np0 = 0, np1 = 0, ni0 = 0, ni1 = 0, n_item = 0;
      bool ok = true;
      Item w;
      auto issue_qk = [&](const int x, uint32_t k_stage) {
        const uint32_t k_lo = k_lo0 + k_stage * (kTileBytes >> 4);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) qk_step(x, k_lo, ks);
        umma_commit(bar(kBarSFull + x));
      };
      // one M tile's share of tile i: O += P V, then S of the next tile (in place of P: the
      // tensor pipe runs its operations in order)
      auto chain = [&](const int x, uint32_t& np_x, const uint32_t ni_x, int i, int n_tiles, uint32_t k_stage,
                       uint32_t v_stage) -> bool {
        // O of the previous item must have been read out before the first PV overwrites it
        if (i == 0 && !mbar_wait(bar(kBarOEmpty + x), (ni_x & 1) ^ 1, abort_flag)) return false;
        if (!mbar_wait(bar(kBarPFull + x), np_x & 1, abort_flag)) return false;
        ++np_x;
        tc_fence_after();
        issue_pv(x, v_stage, i == 0);
        if (i + 1 < n_tiles) {
          issue_qk(x, k_stage);
          if (i + 2 == n_tiles) umma_commit(bar(kBarQEmpty + x));
        } else {
          umma_commit(bar(kBarOFull + x));
        }
        return true;
      };
      while (read_item(n_item, w, ok, false)) {
        ++n_item;
        if (w.n_tiles == 0) continue;
        const bool has_b = w.has_b();
        // S of the first tile for both M tiles
        ok = mbar_wait(bar(kBarQFull + 0), ni0 & 1, abort_flag);
        if (ok && has_b) ok = mbar_wait(bar(kBarQFull + 1), ni1 & 1, abort_flag);
        if (ok) ok = mbar_wait(bar(kBarKReady + tk % KS), (tk / KS) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        issue_qk(0, tk % KS);
        if (w.n_tiles == 1) umma_commit(bar(kBarQEmpty + 0));
        if (has_b) {
          issue_qk(1, tk % KS);
          if (w.n_tiles == 1) umma_commit(bar(kBarQEmpty + 1));
        }
        umma_commit(bar(kBarKEmpty + tk % KS));
        ++tk;
        for (int i = 0; i < w.n_tiles && ok; ++i) {
          const bool next = i + 1 < w.n_tiles;
          const uint32_t k_stage = tk % KS, v_stage = tv % VS;
          if (next) ok = mbar_wait(bar(kBarKReady + k_stage), (tk / KS) & 1, abort_flag);
          if (ok) ok = mbar_wait(bar(kBarVFull + v_stage), (tv / VS) & 1, abort_flag);
          if (ok) ok = chain(0, np0, ni0, i, w.n_tiles, k_stage, v_stage);
          if (ok && has_b) ok = chain(1, np1, ni1, i, w.n_tiles, k_stage, v_stage);
          if (!ok) break;
          umma_commit(bar(kBarVEmpty + v_stage));
          ++tv;
          if (next) {
            umma_commit(bar(kBarKEmpty + k_stage));
            ++tk;
          }
        }
        if (!ok) break;
        ++ni0;
        if (has_b) ++ni1;
      }
      if (!ok) {
        umma_commit(bar(kBarDrain));
        mbar_wait(bar(kBarDrain), 0, abort_flag + 1);
      }
    }
    __syncwarp();
  };
  auto role_rotate_k = [&]() {
    // ------------------------------------------- K tiles re-encoded where they landed
    // A thread owns the same rotary pairs of every tile: 16-byte chunk jj of the low half of a row and
    // chunk jj + PPR of the high half, rows row0, row0 + kRowStep, ...: its eight frequencies never change,
    // and neither does the swizzle (kRowStep is a multiple of 8).  Angles: fp64 once per tile (or per shot, when
    // the keys are stored rotated), then kRowStep positions further by one complex multiplication.
    constexpr int PPR = D / 16;
    constexpr int kRowStep = 32 * kRotateWarps / PPR;
    constexpr int kUnits = kTileN / kRowStep;
    constexpr int RPW = 32 / PPR;                     // rows of one unit in a warp
    static_assert(kRowStep % 8 == 0, "the swizzle of a thread's rows must not change");
    const int lw = warp - kRotateWarp0;
    const int jj = lane % PPR, row0 = lw * RPW + lane / PPR;
    const int map_row = (lane / RPW) * kRowStep + lw * RPW + lane % RPW;     // the row whose map entry this lane loads
    const uint32_t off_lo = (jj / 8) * 16384u + row0 * 128u + (((jj & 7) ^ (row0 & 7)) << 4);
    const uint32_t off_hi = ((jj + PPR) / 8) * 16384u + row0 * 128u + ((((jj + PPR) & 7) ^ (row0 & 7)) << 4);
    const double* theta = p.theta + jj * 8;
    const bool per_shot = p.k_pos_mode == 1;          // the angle is that of the shot's first position
    float2 step_c[4], step_s[4];                      // (cos, sin) of kRowStep positions, two frequencies each
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      rope_sincos((double)kRowStep, theta[2 * e], &step_s[e].x, &step_c[e].x);
      rope_sincos((double)kRowStep, theta[2 * e + 1], &step_s[e].y, &step_c[e].y);
    }
    float2 c2[4], s2[4];                              // (cos, sin) of the current row
    auto set_angles = [&](double delta) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        rope_sincos_fast(delta, theta[2 * e], &s2[e].x, &c2[e].x);
        rope_sincos_fast(delta, theta[2 * e + 1], &s2[e].y, &c2[e].y);
      }
    };
    auto rotate_unit = [&](unsigned char* kt, int u, bool step) {
      uint4* lo = reinterpret_cast<uint4*>(kt + off_lo + u * kRowStep * 128u);
      uint4* hi = reinterpret_cast<uint4*>(kt + off_hi + u * kRowStep * 128u);
      const uint4 xl = *lo, yl = *hi;
      const uint32_t xw[4] = {xl.x, xl.y, xl.z, xl.w}, yw[4] = {yl.x, yl.y, yl.z, yl.w};
      uint32_t xo[4], yo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 x = make_float2(__uint_as_float(xw[e] << 16), __uint_as_float(xw[e] & 0xffff0000u));
        const float2 y = make_float2(__uint_as_float(yw[e] << 16), __uint_as_float(yw[e] & 0xffff0000u));
        const float2 ns = make_float2(-s2[e].x, -s2[e].y);
        const float2 xr = __ffma2_rn(y, ns, __fmul2_rn(x, c2[e]));
        const float2 yr = __ffma2_rn(x, s2[e], __fmul2_rn(y, c2[e]));
        xo[e] = pack_bf16x2(xr.x, xr.y);
        yo[e] = pack_bf16x2(yr.x, yr.y);
        if (step) {
          const float2 c = __ffma2_rn(ns, step_s[e], __fmul2_rn(c2[e], step_c[e]));
          s2[e] = __ffma2_rn(c2[e], step_s[e], __fmul2_rn(s2[e], step_c[e]));
          c2[e] = c;
        }
      }
      *lo = make_uint4(xo[0], xo[1], xo[2], xo[3]);
      *hi = make_uint4(yo[0], yo[1], yo[2], yo[3]);
    };
    uint32_t tk = 0;
    bool ok = true;
    Item w;
    for (uint32_t n_item = 0; ok && read_item(n_item, w, ok, true); ++n_item) {
      const int* omap = p.off_map + (long long)w.b * p.ctx_cap;
      auto first_of = [&](int i) -> int {           // first position of the shot that map_row of tile i lies in
        const long long pos = (long long)(w.ctx_begin + i) * kTileN + map_row;
        return per_shot && i < w.n_ctx && pos < p.ctx_cap ? omap[pos] : 0;
      };
      int first = first_of(0), first_cur = -1;
      for (int i = 0; i < w.n_tiles; ++i, ++tk) {
        const uint32_t sk = tk % KS;
        unsigned char* kt = base_ptr + SM::kOffK + sk * kTileBytes;
        const bool ctx = i < w.n_ctx;               // (the probe's own keys were rotated by the prep kernel)
        const int first_next = first_of(i + 1);
        if (ctx && !per_shot) set_angles((double)((long long)(w.ctx_begin + i) * kTileN + row0));
        ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarKFull + sk), (tk / KS) & 1, abort_flag));
        if (!ok) break;
        if (ctx && !per_shot) {
#pragma unroll
          for (int u = 0; u < kUnits; ++u) rotate_unit(kt, u, u + 1 < kUnits);
        } else if (ctx) {
#pragma unroll 2
          for (int u = 0; u < kUnits; ++u) {
            const int o = __shfl_sync(0xffffffffu, first, u * RPW + lane / PPR);
            if (o != first_cur) {
              set_angles((double)o);
              first_cur = o;
            }
            rotate_unit(kt, u, false);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kBarKRot + sk));
        first = first_next;
      }
    }
  };
  auto role_gather = [&]() {
    // ----------------------------------------------- V (fused: K, too) tiles straight from the pool, stitched by TMA
    // Eq. 7 corrects K only, so V needs no assembled copy.  The 128 context positions of a tile map
    // to a few runs of consecutive pool rows (one per selected shot the tile touches): the lanes look
    // the positions up and mark where a run ends; every run is brought as one or two power-of-two boxes
    // (maps with 128, 64, ..., 1-row boxes over the pool; a box may start at any row, its shared-memory
    // address only has to be 128-byte aligned), one box per lane, all found before the stage is waited
    // for.  Positions beyond the context take rows outside the pool, which arrive as zeros: their P is exactly zero,
    // but 0 times what the next shot of the pool holds need not be.  The probe's own tokens are one run of
    // the own-token tensor.
    const bool is_k = FUSED && warp != kGatherWarp;
    int* rows_s = reinterpret_cast<int*>(base_ptr + SM::kOffRows + (is_k ? 512 : 0));
    const uint32_t n_st = is_k ? KS : VS;
    const uint32_t tiles0 = base + (is_k ? SM::kOffK : SM::kOffV);
    const uint32_t full0 = bar(is_k ? kBarKFull : kBarVFull), empty0 = bar(is_k ? kBarKEmpty : kBarVEmpty);
    const PoolMaps* maps = is_k ? &kmaps : &vmaps;
    const CUtensorMap* own_map = is_k ? &tm_kown : &tm_vown;
    uint32_t sv = 0, phase = 0;                  // stage and parity of tile tv
    uint32_t tv = 0;
    bool ok = true;
    Item w;
    for (uint32_t n_item = 0; ok && read_item(n_item, w, ok, true); ++n_item) {
      for (int i = 0; i < w.n_tiles; ++i, ++tv, phase ^= (sv + 1 == n_st), sv = sv + 1 == n_st ? 0 : sv + 1) {
        const uint32_t v_dst = tiles0 + sv * kTileBytes;
        const uint32_t full = full0 + 8u * sv;
        if (i >= w.n_ctx) {
          // own tokens: one tiled box (rows beyond the last own token arrive as zeros)
          if (lane == 0) {
            ok = mbar_wait(empty0 + 8u * sv, phase ^ 1, abort_flag);
            if (ok) {
              mbar_arrive_expect_tx(full, kTileBytes);
#pragma unroll
              for (int s2 = 0; s2 < SUB; ++s2)
                tma_load_4d(v_dst + s2 * 16384u, own_map, full, s2 * 64, w.g,
                            (w.own_begin + i - w.n_ctx) * kTileN, w.outer_own);
            }
          }
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
          if (!ok) break;
          continue;
        }
        // pool row of positions lane, lane + 32, lane + 64, lane + 96 of the tile (looked up while the
        // stage may still be in use)
        const long long pos0 = (long long)(w.ctx_begin + i) * kTileN;
        const long long L_all = p.ctx_cap;            // (row map entries beyond a query's context are -1)
        int r[4];
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          const long long pos = pos0 + lane + 32 * q4;
          r[q4] = pos < L_all ? p.row_map[(long long)w.b * p.ctx_cap + pos] : -1;
        }
        // the number of valid positions of the tile: they form a prefix (valid positions are 0 .. L-1)
        unsigned valid_mask[4];
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) valid_mask[q4] = __ballot_sync(0xffffffffu, r[q4] >= 0);
        const int n_valid = __popc(valid_mask[0]) + __popc(valid_mask[1]) + __popc(valid_mask[2]) + __popc(valid_mask[3]);
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          const int pidx = lane + 32 * q4;
          if (pidx >= n_valid) r[q4] = pidx - 2 * kTileN;       // one run of rows in front of the pool: zeros
        }
        __syncwarp();
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) rows_s[lane + 32 * q4] = r[q4];
        // a run ends after position pidx when the next position is not the next pool row
        unsigned brk[4];
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          int nxt = __shfl_down_sync(0xffffffffu, r[q4], 1);
          const int wrap = __shfl_sync(0xffffffffu, q4 < 3 ? r[q4 + 1 < 4 ? q4 + 1 : 3] : 0, 0);
          if (lane == 31) nxt = wrap;
          const bool last = lane == 31 && q4 == 3;
          brk[q4] = __ballot_sync(0xffffffffu, last || nxt != r[q4] + 1);
        }
        // the run ends as one 128-bit mask in every lane; lane j then finds the j-th box on its own.
        // A run of n rows takes the largest power-of-two box that fits, once from its first row and,
        // unless n is that power of two, once more ending at its last row: the two overlap, both write
        // the same values there, and no run needs more than two copy instructions (the copy engine's
        // time goes with the number of instructions, not with the bytes)
        __syncwarp();
        int my_pidx = -1, my_row = 0, my_lg = 0, n_boxes = 0;
        uint32_t tile_bytes = 0;                 // what the boxes deliver in all (overlaps are copied twice)
        {
          int pidx = 0;
          while (pidx < kTileN) {
            int e = pidx;                       // end of the run that starts at pidx: first set bit at or after it
            for (;;) {
              const unsigned word = (e < 32 ? brk[0] : e < 64 ? brk[1] : e < 96 ? brk[2] : brk[3]) >> (e & 31);
              if (word != 0) { e += __ffs(word) - 1; break; }
              e = (e | 31) + 1;
            }
            const int n = e - pidx + 1;
            const int lg = 31 - __clz(n);        // the largest power-of-two box that fits
            if (n_boxes == lane) { my_pidx = pidx; my_lg = lg; }
            ++n_boxes;
            if (n > (1 << lg)) {                 // the rest of the run: the same box once more, ending at the run's end
              if (n_boxes == lane) { my_pidx = e + 1 - (1 << lg); my_lg = lg; }
              ++n_boxes;
            }
            tile_bytes += (n > (1 << lg) ? 2u : 1u) * ((uint32_t)SUB << (lg + 7));
            pidx = e + 1;
          }
        }
        if (my_pidx >= 0) my_row = rows_s[my_pidx];
        // (tiles of more than 32 boxes - many one-token shots - take further rounds of the same walk)
        if (lane == 0) {
          ok = mbar_wait(empty0 + 8u * sv, phase ^ 1, abort_flag);
          if (ok) mbar_arrive_expect_tx(full, tile_bytes);
        }
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) break;
        const int layer = p.layer_begin + w.l;
        if (my_pidx >= 0) {
#pragma unroll
          for (int s2 = 0; s2 < SUB; ++s2)
            tma_load_4d(v_dst + s2 * 16384u + (uint32_t)my_pidx * 128u, &maps->m[my_lg], full, s2 * 64,
                        w.g, my_row, layer);
        }
        for (int round = 1; round * 32 < n_boxes; ++round) {      // rare: more than 32 boxes in the tile
          int pidx = 0, idx = 0, bp = -1, bl = 0;
          while (pidx < kTileN) {
            int e = pidx;
            for (;;) {
              const unsigned word = (e < 32 ? brk[0] : e < 64 ? brk[1] : e < 96 ? brk[2] : brk[3]) >> (e & 31);
              if (word != 0) { e += __ffs(word) - 1; break; }
              e = (e | 31) + 1;
            }
            const int n = e - pidx + 1;
            const int lg = 31 - __clz(n);
            if (idx == round * 32 + lane) { bp = pidx; bl = lg; }
            ++idx;
            if (n > (1 << lg)) {
              if (idx == round * 32 + lane) { bp = e + 1 - (1 << lg); bl = lg; }
              ++idx;
            }
            pidx = e + 1;
          }
          if (bp >= 0) {
            const int brow = rows_s[bp];
#pragma unroll
            for (int s2 = 0; s2 < SUB; ++s2)
              tma_load_4d(v_dst + s2 * 16384u + (uint32_t)bp * 128u, &maps->m[bl], full, s2 * 64, w.g,
                          brow, layer);
          }
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) {
      // gave up: let the copies already in flight land before the CTA retires
      for (uint32_t t = tv > n_st ? tv - n_st : 0; t < tv; ++t)
        mbar_wait(full0 + 8u * (t % n_st), (t / n_st) & 1, abort_flag + 1);
    }
    __syncwarp();
  };
  auto role_softmax = [&]() {
    // ---------------------------------------------------- softmax + read-out of O
    const int x = (warp - kSoftmaxWarp0) >> 2;     // 0: M tile A, 1: M tile B
    const int quarter = warp & 3;                  // TMEM lanes this warp may touch
    const int r = quarter * 32 + lane;             // row of the M tile
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t s_addr = tmem_base + lane_addr + kTmemS + x * kTileN;
    const uint32_t o_addr = tmem_base + lane_addr + kTmemO + x * 128;
    uint32_t ns = 0, ni = 0;
    bool ok = true;
    auto warp_arrive = [&](uint32_t b) {             // this warp's share of a barrier that four warps complete
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b);
    };
    for (uint32_t n_item = 0; ok; ++n_item) {
      // (the item is read where it lies: its fields would cost registers over the whole tile loop)
      const uint32_t islot = n_item % kItems;
      ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarItemFull + islot), (n_item / kItems) & 1, abort_flag));
      if (!ok) break;
      const Item& w = items[islot];
      const int n_tiles = w.n_tiles;
      if (n_tiles < 0) break;
      if (x == 0 || w.has_b()) {
        const int mt = 2 * w.mp + x;
        const int m = mt * kTileM + r;               // row of the unit: token m / G, head m % G
        const int t_row = div_g(p, m);
        float m_used = kNegSentinel, l_sum = 0.f;
        // columns below a limit are visible, 128 fewer with every tile: context keys before L_j, own keys up to the row's token
        const int n_ctx = w.n_ctx;
        const int ctx_limit = w.Lj - w.ctx_begin * kTileN;
        const int own_limit = p.To - p.Tq + min(t_row, p.Tq - 1) + 1 + (n_ctx - w.own_begin) * kTileN;
        for (int i = 0; i < n_tiles; ++i, ++ns) {
          ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarSFull + x), ns & 1, abort_flag));
          if (!ok) break;
          tc_fence_after();
          float s[kTileN];
          if constexpr (FUSED) tmem_ld4x32(s_addr, reinterpret_cast<uint32_t*>(s));
          else tmem_ld128(s_addr, reinterpret_cast<uint32_t*>(s));

          // mask: only the last context tile and the own-token tiles can hide anything (limit <= 0: all of it)
          const int limit = (i < n_ctx ? ctx_limit : own_limit) - i * kTileN;
          if (__any_sync(0xffffffffu, limit < kTileN)) {
#pragma unroll
            for (int cidx = 0; cidx < kTileN; ++cidx) s[cidx] = cidx < limit ? s[cidx] : -INFINITY;
          }
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int cidx = 0; cidx < kTileN; cidx += 8) {
#pragma unroll
            for (int u = 0; u < 4; ++u) mx[u] = fmax3(mx[u], s[cidx + 2 * u], s[cidx + 2 * u + 1]);
          }
          const float tile_max = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.scale_log2;
          float alpha = 1.f;
          const bool need = tile_max > m_used + kRescaleThreshold;
          if (need) {
            alpha = exp2f(m_used - tile_max);
            m_used = tile_max;
            l_sum *= alpha;
          }
          // P = 2^(s * scale - m) as packed bf16 back into the S columns (two keys per column);
          // scale-and-shift and the row sum run two columns per instruction (packed fp32)
          const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
          const float2 neg_m2 = make_float2(-m_used, -m_used);
          float2 part[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
          auto exp_pair = [&](int c2) -> uint32_t {
            const float2 xs = __ffma2_rn(make_float2(s[2 * c2], s[2 * c2 + 1]), scale2, neg_m2);
            const float2 e = make_float2(ex2_approx(xs.x), ex2_approx(xs.y));
            part[c2 & 3] = __fadd2_rn(part[c2 & 3], e);
            return pack_bf16x2(e.x, e.y);
          };
          if constexpr (FUSED) {
            // 32 keys at a time: their 16 packed columns are stored while the next ones are computed
#pragma unroll
            for (int c0 = 0; c0 < kTileN / 2; c0 += 16) {
              uint32_t pk[16];
#pragma unroll
              for (int c = 0; c < 16; ++c) pk[c] = exp_pair(c0 + c);
              tmem_st16_nowait(s_addr + c0, pk);
            }
            tmem_st_wait();
          } else {
            // the packed pair c2 goes into the register that held score c2 (already consumed:
            // c2 <= 2 c2), so the row never needs more than its 128 registers
            uint32_t* pk = reinterpret_cast<uint32_t*>(s);
#pragma unroll
            for (int c2 = 0; c2 < kTileN / 2; ++c2) pk[c2] = exp_pair(c2);
            tmem_st64(s_addr, pk);
          }
          const float2 tot = __fadd2_rn(__fadd2_rn(part[0], part[1]), __fadd2_rn(part[2], part[3]));
          l_sum += tot.x + tot.y;
          if (i > 0 && __any_sync(0xffffffffu, need)) {
            // S(i) is complete, so PV(i-1), issued before it, is complete too; PV(i) waits for
            // the arrival below: O is quiescent here.
#pragma unroll
            for (int q4 = 0; q4 < D / 32; ++q4) {
              float o[32];
              tmem_ld32(o_addr + q4 * 32, reinterpret_cast<uint32_t*>(o));
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] *= alpha;
              tmem_st32(o_addr + q4 * 32, reinterpret_cast<const uint32_t*>(o));
            }
          }
          warp_arrive(bar(kBarPFull + x));
        }
        if (!ok) break;
        const bool row_ok = m < p.Tq * p.G;
        if (n_tiles == 0) {
          // nothing of this M pair falls into the piece: a neutral partial (a whole unit is never empty)
          float4* otile = reinterpret_cast<float4*>(p.o_part) + (w.slot * 2 + x) * ((long long)(D / 4) * kTileM) + r;
#pragma unroll
          for (int c4 = 0; c4 < D / 4; ++c4) otile[c4 * kTileM] = make_float4(0.f, 0.f, 0.f, 0.f);
          float* ml = p.ml_part + ((long long)(w.slot * 2 + x) * kTileM + r) * 2;
          ml[0] = kNegSentinel;
          ml[1] = 0.f;
        } else {
          ok = __all_sync(0xffffffffu, mbar_wait(bar(kBarOFull + x), ni & 1, abort_flag));
          if (!ok) break;
          tc_fence_after();
          if (w.whole()) {
            // The piece covers the unit: normalise and store the final rows.  A thread owns a
            // row, and rows are far apart in the output, so a direct store would touch 32 lines
            // per instruction; instead the warp passes 64 columns at a time through its staging
            // area (16-byte chunks swizzled by the row) and writes four rows' 128-byte segments
            // per instruction.
            const float inv = 1.f / l_sum;
            const long long bpj = w.outer_own;
            unsigned char* stg = base_ptr + SM::kOffStage + (warp - kSoftmaxWarp0) * SM::kStageBytes;
            const int sub = lane >> 3, ch = lane & 7;            // read-back: row 4 j + sub, chunk ch
            const int m0 = mt * kTileM + quarter * 32;
            if constexpr (FUSED) {
              // (no staging area in the fused variant's shared-memory plan: one row per thread)
              const int hq = w.g * p.G + m - t_row * p.G;
              __nv_bfloat16* dst = p.out + (((bpj * p.Tq + t_row) * p.Hq) + hq) * (long long)D;
#pragma unroll
              for (int q4 = 0; q4 < D / 32; ++q4) {
                float o[32];
                tmem_ld32(o_addr + q4 * 32, reinterpret_cast<uint32_t*>(o));
                if (q4 == D / 32 - 1) warp_arrive(bar(kBarOEmpty + x));
                if (row_ok) {
#pragma unroll
                  for (int e = 0; e < 32; e += 8) {
                    float v8[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v8[u] = o[e + u] * inv;
                    *reinterpret_cast<uint4*>(dst + q4 * 32 + e) = bf16x8_pack(v8);
                  }
                }
              }
            } else {
#pragma unroll
            for (int h = 0; h < D / 64; ++h) {
              float o[64];
              tmem_ld32(o_addr + h * 64, reinterpret_cast<uint32_t*>(o));
              tmem_ld32(o_addr + h * 64 + 32, reinterpret_cast<uint32_t*>(o + 32));
              if (h == D / 64 - 1) warp_arrive(bar(kBarOEmpty + x));     // O is in registers: the next item may overwrite it
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                float v8[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v8[u] = o[c * 8 + u] * inv;
                *reinterpret_cast<uint4*>(stg + lane * 128 + ((c ^ (lane & 7)) << 4)) = bf16x8_pack(v8);
              }
              __syncwarp();
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const int row = 4 * j + sub;
                const int mm = m0 + row;
                const uint4 v = *reinterpret_cast<const uint4*>(stg + row * 128 + ((ch ^ (row & 7)) << 4));
                if (mm < p.Tq * p.G) {
                  const int tt = div_g(p, mm), hq = w.g * p.G + mm - tt * p.G;
                  __nv_bfloat16* dst = p.out + (((bpj * p.Tq + tt) * p.Hq) + hq) * (long long)D;
                  *reinterpret_cast<uint4*>(dst + h * 64 + ch * 8) = v;
                }
              }
              __syncwarp();
            }
            }
            if (row_ok && p.lse != nullptr) {
              const int hh = m - t_row * p.G, hq = w.g * p.G + hh;
              p.lse[(bpj * p.Hq + hq) * p.Tq + t_row] = (m_used + log2f(l_sum)) * kLn2;
            }
          } else {
            // un-normalised partial, four columns of 128 rows at a time ([D/4][128][4] per M tile):
            // a warp's 32 rows are 512 contiguous bytes per store
            float4* otile = reinterpret_cast<float4*>(p.o_part) + (w.slot * 2 + x) * ((long long)(D / 4) * kTileM) + r;
#pragma unroll
            for (int q4 = 0; q4 < D / 32; ++q4) {
              float o[32];
              tmem_ld32(o_addr + q4 * 32, reinterpret_cast<uint32_t*>(o));
              if (q4 == D / 32 - 1) warp_arrive(bar(kBarOEmpty + x));
#pragma unroll
              for (int e = 0; e < 32; e += 4)
                otile[(q4 * 8 + e / 4) * kTileM] = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
            }
            float* ml = p.ml_part + ((long long)(w.slot * 2 + x) * kTileM + r) * 2;
            ml[0] = m_used;
            ml[1] = l_sum;
          }
          ++ni;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kBarItemEmpty + islot));
    }
  };

  // registers go where they are needed, one warpgroup at a time
  if (warp < 4) {
    regs_lower<FUSED ? kFusedRegsIssue : kRegsIssue>();
    if (warp == 0) role_tma();
    else if (FUSED ? warp != 1 : VPOOL && warp == kGatherWarp) role_gather();
    else if (warp == 1) role_mma();
  } else if (!FUSED || warp < kRotateWarp0) {
    regs_raise<FUSED ? kFusedRegsSoftmax : kRegsSoftmax>();
    role_softmax();
  } else if constexpr (FUSED) {
    regs_lower<kFusedRegsRotate>();
    role_rotate_k();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
  if (threadIdx.x == 0 && *abort_flag != 0) ads_set_status(p.status, ADAPSHOT_ETIMEOUT);
}

struct CombineParams {
  const Sched* sched;
  const float* o_part;
  const float* ml_part;
  __nv_bfloat16* out;   // [B][nl][P][Tq][Hq][D]
  float* lse;           // [B][nl][P][Hq][Tq] or null
  int Tq, Hq, G, n_mp;
  int units;                  // of the grid (units, groups of rows, column steps); the blocks beyond them:
  AdsEntropyJob ent;          // the entropy's second step, a block per query
};

constexpr int kCombineRows = 8;      // rows per warp
constexpr int kCombineSteps = 2;     // 16-column steps per warp (blockIdx.z covers the others)

// Block x merges the x-th of the units that a range boundary cut (listed by the schedule block, so that
// nothing has to be searched for here).  Latency- and L2-bound: one query of one layer (26 MB of partials)
// took 14.6 us when every block searched the schedule and merged piece after piece, 8.8 us now; in front of
// a cache of 12 K tokens, cut into eighteen pieces per unit, 19.4 and 7.4 us.  A warp merges 8 rows: lane = (row r_sub, 4-column chunk c_sub of the 16 columns of one step),
// so that a load is 8 rows x 16 bytes contiguous per chunk in the partial layout ([D/4][128 rows][4] per
// M tile) and a store fills one 32-byte sector per row.
template <int D>
__global__ void __launch_bounds__(256) attn_combine_kernel(const __grid_constant__ CombineParams p) {
  ads_dependency_wait();
  if ((int)blockIdx.x >= p.units) {
    __shared__ float sh_h[kMaxProbes];               // (a group is a query's probes)
    const int group = (((int)blockIdx.x - p.units) * (int)gridDim.y + (int)blockIdx.y) * (int)gridDim.z + (int)blockIdx.z;
    if (group < p.ent.R / p.ent.rows_per_group)
      ent_finish_block(p.ent.partial, p.ent.n_split, p.ent.R, p.ent.rows_per_group, p.ent.tau, p.ent.H, p.ent.first_ok, group, sh_h);
    return;
  }
  const Sched* sc = p.sched;
  if (blockIdx.x >= sc->n_cut) return;
  const Sched::Cut c = sc->cut[blockIdx.x];
  const int lane = threadIdx.x & 31;
  const int r_sub = lane & 7, c_sub = lane >> 3;
  const int m = (blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kCombineRows + r_sub;
  if (m >= p.Tq * p.G) return;
  const int mt = m / kTileM, r = m % kTileM, mp = mt >> 1, x = mt & 1;
  const int t = m / p.G, hh = m % p.G, h = c.g * p.G + hh;
  const long long bpj = c.bpj;
  auto slot_tile = [&](int i) -> long long {        // tile of piece i
    return ((long long)(2 * (c.gang + i) + (i == 0 ? c.which : 0)) * p.n_mp + mp) * 2 + x;
  };
  const float4* o4 = reinterpret_cast<const float4*>(p.o_part);
  const int it0 = blockIdx.z * kCombineSteps;
  float4 acc[kCombineSteps];
#pragma unroll
  for (int it = 0; it < kCombineSteps; ++it) acc[it] = make_float4(0.f, 0.f, 0.f, 0.f);
  float M = kNegSentinel, lsum = 0.f;
  // the loads of four pieces are issued before any is merged (running maximum, one pass)
  for (int i0 = 0; i0 < c.n; i0 += 4) {
    float2 ml[4];
    float4 v[4][kCombineSteps];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool use = i0 + u < c.n;
      const long long tile = slot_tile(use ? i0 + u : 0);
      ml[u] = use ? *reinterpret_cast<const float2*>(p.ml_part + (tile * kTileM + r) * 2) : make_float2(kNegSentinel, 0.f);
#pragma unroll
      for (int it = 0; it < kCombineSteps; ++it)
        v[u][it] = use ? o4[(tile * (D / 4) + (it0 + it) * 4 + c_sub) * kTileM + r] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float m_new = fmaxf(fmaxf(M, fmaxf(ml[0].x, ml[1].x)), fmaxf(ml[2].x, ml[3].x));
    const float keep = exp2f(M - m_new);
    M = m_new;
    lsum *= keep;
#pragma unroll
    for (int it = 0; it < kCombineSteps; ++it) {
      acc[it].x *= keep; acc[it].y *= keep; acc[it].z *= keep; acc[it].w *= keep;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float wgt = exp2f(ml[u].x - M);
      lsum += ml[u].y * wgt;
#pragma unroll
      for (int it = 0; it < kCombineSteps; ++it) {
        acc[it].x += v[u][it].x * wgt; acc[it].y += v[u][it].y * wgt;
        acc[it].z += v[u][it].z * wgt; acc[it].w += v[u][it].w * wgt;
      }
    }
  }
  const float inv = 1.f / lsum;
  __nv_bfloat16* dst = p.out + (((bpj * p.Tq + t) * p.Hq) + h) * (long long)D;
#pragma unroll
  for (int it = 0; it < kCombineSteps; ++it) {
    uint2 packed;
    packed.x = pack_bf16x2(acc[it].x * inv, acc[it].y * inv);
    packed.y = pack_bf16x2(acc[it].z * inv, acc[it].w * inv);
    *reinterpret_cast<uint2*>(dst + ((it0 + it) * 4 + c_sub) * 4) = packed;
  }
  if (p.lse != nullptr && c_sub == 0 && blockIdx.z == 0)
    p.lse[(bpj * p.Hq + h) * p.Tq + t] = (M + log2f(lsum)) * kLn2;
}

// Self-test of the bounded wait every pipeline barrier uses: warp 0 waits (with a limit of about a
// millisecond) on a barrier that nothing will ever complete, gives up, raises the CTA's abort flag
// and reports ADAPSHOT_ETIMEOUT; warp 1 waits on the same barrier with the long limit and must
// return as soon as it sees the flag.  The kernel ends normally: the context stays usable.
__global__ void __launch_bounds__(64) wait_timeout_selftest_kernel(int32_t* status, long long* cycles) {
  __shared__ __align__(8) unsigned long long barmem;
  __shared__ int abort_flag[2];
  const uint32_t b = smem_u32(&barmem);
  if (threadIdx.x == 0) {
    mbar_init(b, 1);
    abort_flag[0] = abort_flag[1] = 0;
    mbar_fence_init();
  }
  __syncthreads();
  const long long t0 = clock64();
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait_limit(b, 0, abort_flag, 2000000ll);
  if (threadIdx.x == 32) ok = mbar_wait(b, 0, abort_flag);
  if ((threadIdx.x & 31) == 0) cycles[threadIdx.x >> 5] = ok ? -1 : clock64() - t0;
  __syncthreads();
  if (threadIdx.x == 0 && abort_flag[0] != 0) ads_set_status(status, ADAPSHOT_ETIMEOUT);
}

// ----------------------------------------------------------------- host side
// bf16 tensor, innermost dim contiguous, 128-byte swizzle, zero fill outside the bounds
bool make_map(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
              const uint32_t* box) {
  return ads_make_bf16_map(m, base, rank, dims, strides_bytes, box);
}

// Optional timing of the main kernel alone (adapshot_profile): two events around its launch.
bool g_profile = false;
bool g_profile_valid = false;
cudaEvent_t g_profile_ev[2] = {nullptr, nullptr};

struct AttnPlan {
  int n_mt, n_mp, gang;
  size_t off_qrot, off_kqrot, off_sched, off_opart, off_ml, off_rowmap, off_offmap, total;
};

// Own tokens beyond the query rows, and a per-query shot count on the device (decode calls).
struct AttnExtra {
  int To = 0;                        // 0: as many own tokens as query rows
  const int32_t* nshots_dev = nullptr;
  AdsPass pass = {};                 // what a pass in one call shares
};

// What the fused variant reads instead of an assembled cache.
struct FusedSrc {
  const adapshot_pool_t* pool;
  const int32_t* sel_idx;
  int layer_begin;
};

// The gang (CTAs that walk the same K/V tiles, one M pair each per round) is the number of
// M pairs when that is at most kMaxGang, else the M pairs are dealt out in rounds.
AttnPlan make_plan(const adapshot_model_t* model, int B, int P, int Tq, int nl, long long map_ctx_cap = 0, int To = 0) {
  if (To < Tq) To = Tq;
  AttnPlan pl;
  const int G = model->n_q_heads / model->n_kv_heads;
  const int D = model->head_dim;
  pl.n_mt = (Tq * G + kTileM - 1) / kTileM;
  pl.n_mp = (pl.n_mt + 1) / 2;
  const int rounds = (pl.n_mp + kMaxGang - 1) / kMaxGang;
  pl.gang = (pl.n_mp + rounds - 1) / rounds;
  const size_t slots = (size_t)2 * kMaxCtas * pl.n_mp;     // two cut pieces per gang at most
  size_t off = 0;
  pl.off_qrot = off;  off += ads_round_up((size_t)B * nl * P * Tq * model->n_q_heads * D * 2, 256);
  pl.off_kqrot = off; off += ads_round_up((size_t)B * nl * P * To * model->n_kv_heads * D * 2, 256);
  pl.off_sched = off; off += ads_round_up(sizeof(Sched), 256);
  pl.off_opart = off; off += ads_round_up(slots * 2 * kTileM * D * 4, 256);
  pl.off_ml = off;    off += ads_round_up(slots * 2 * kTileM * 2 * 4, 256);
  pl.off_rowmap = off; off += ads_round_up((size_t)B * map_ctx_cap * 4, 256);
  pl.off_offmap = off; off += ads_round_up((size_t)B * map_ctx_cap * 4, 256);
  pl.total = off;
  return pl;
}

bool attn_shape_ok(const adapshot_model_t* m) {
  return (m->head_dim == 64 || m->head_dim == 128) && m->n_kv_heads > 0 && m->n_q_heads > 0 &&
         m->n_q_heads % m->n_kv_heads == 0;
}

template <int D>
int launch_attn(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx, int64_t ctx_cap,
                const int64_t* ctx_off, int B, int k, const int32_t* probe_nshots, int P, const void* q,
                const void* kq, const void* vq, int Tq, int nl, void* out, float* lse, const AttnPlan& pl,
                void* ws, int32_t* status, cudaStream_t st, const FusedSrc* fused = nullptr,
                int mode = kModeCache, AttnExtra extra = AttnExtra()) {
  const int To = extra.To > Tq ? extra.To : Tq;
  const int Hq = model->n_q_heads, Hkv = model->n_kv_heads, G = Hq / Hkv;
  unsigned char* wsb = static_cast<unsigned char*>(ws);
  __nv_bfloat16* q_rot = reinterpret_cast<__nv_bfloat16*>(wsb + pl.off_qrot);
  __nv_bfloat16* kq_rot = reinterpret_cast<__nv_bfloat16*>(wsb + pl.off_kqrot);
  Sched* sched = reinterpret_cast<Sched*>(wsb + pl.off_sched);
  float* o_part = reinterpret_cast<float*>(wsb + pl.off_opart);
  float* ml_part = reinterpret_cast<float*>(wsb + pl.off_ml);

  const int n_sm = ads_sm_count();
  if (n_sm <= 0) return ADAPSHOT_ECUDA;
  const int n_cta = n_sm < kMaxCtas ? n_sm : kMaxCtas;
  const int n_gangs = n_cta / pl.gang > 0 ? n_cta / pl.gang : 1;

  // ---- tensor maps
  CUtensorMap tm_q, tm_kctx, tm_vctx, tm_kown, tm_vown;
  {
    const uint64_t dims[3] = {(uint64_t)D, (uint64_t)Tq * G, (uint64_t)B * nl * P * Hkv};
    const uint64_t str[2] = {(uint64_t)D * 2, (uint64_t)Tq * G * D * 2};
    const uint32_t box[3] = {64, (uint32_t)kTileM, 1};
    if (!make_map(&tm_q, q_rot, 3, dims, str, box)) return ADAPSHOT_ECUDA;
  }
  {
    const uint64_t dims[4] = {(uint64_t)D, (uint64_t)Hkv, (uint64_t)ctx_cap, (uint64_t)B * nl};
    const uint64_t str[3] = {(uint64_t)D * 2, (uint64_t)Hkv * D * 2, (uint64_t)ctx_cap * Hkv * D * 2};
    const uint32_t box[4] = {64, 1, (uint32_t)kTileN, 1};
    tm_kctx = tm_q;                    // (a map the mode never uses: its loader warps read the pool)
    tm_vctx = tm_q;
    if (mode != kModeFused && !make_map(&tm_kctx, k_ctx, 4, dims, str, box)) return ADAPSHOT_ECUDA;
    if (mode == kModeCache && !make_map(&tm_vctx, v_ctx, 4, dims, str, box)) return ADAPSHOT_ECUDA;
  }
  {
    const uint64_t dims[4] = {(uint64_t)D, (uint64_t)Hkv, (uint64_t)To, (uint64_t)B * nl * P};
    const uint64_t str[3] = {(uint64_t)D * 2, (uint64_t)Hkv * D * 2, (uint64_t)To * Hkv * D * 2};
    const uint32_t box[4] = {64, 1, (uint32_t)kTileN, 1};
    if (!make_map(&tm_kown, kq_rot, 4, dims, str, box)) return ADAPSHOT_ECUDA;
    if (!make_map(&tm_vown, vq, 4, dims, str, box)) return ADAPSHOT_ECUDA;
  }
  PoolMaps vmaps, kmaps;
  for (int e = 0; e < 8; ++e) vmaps.m[e] = kmaps.m[e] = tm_q;       // (unused where nothing comes from the pool)
  if (mode != kModeCache) {
    // the pool's V (fused: K, too) with boxes of 1, 2, ..., 128 rows (the layout of the cache maps, over the pool)
    const uint64_t pt = (uint64_t)fused->pool->pool_tokens;
    const uint64_t dims[4] = {(uint64_t)D, (uint64_t)Hkv, pt, (uint64_t)model->n_layers};
    const uint64_t str[3] = {(uint64_t)D * 2, (uint64_t)Hkv * D * 2, pt * Hkv * D * 2};
    for (int e = 0; e < 8; ++e) {
      const uint32_t box[4] = {64, 1, 1u << e, 1};
      if (!make_map(&vmaps.m[e], fused->pool->v, 4, dims, str, box)) return ADAPSHOT_ECUDA;
      if (mode == kModeFused && !make_map(&kmaps.m[e], fused->pool->k, 4, dims, str, box)) return ADAPSHOT_ECUDA;
    }
  }

  // ---- rotate Q and the probe's own K, write the schedule and, for K or V from the pool, the row map
  int* row_map = reinterpret_cast<int*>(wsb + pl.off_rowmap);
  int* off_map = reinterpret_cast<int*>(wsb + pl.off_offmap);
  PrepParams pp;
  pp.ent = extra.pass.ent != nullptr ? *extra.pass.ent : AdsEntropyJob{};
  pp.map = RowMapParams{};
  pp.map_blocks = 0;
  if (fused != nullptr) {
    RowMapParams& rm = pp.map;
    rm.ctx_off = reinterpret_cast<const long long*>(ctx_off);
    rm.sel_idx = fused->sel_idx;
    rm.shot_off = reinterpret_cast<const long long*>(fused->pool->shot_off);
    rm.row_map = row_map;
    rm.off_map = mode == kModeFused && model->k_pos_mode == 1 ? off_map : nullptr;
    rm.ctx_cap = ctx_cap;
    rm.B = B; rm.k = k; rm.n_shots = fused->pool->n_shots;
    pp.map_blocks = (int)(((long long)B * k + 7) / 8);
  }
  pp.q = static_cast<const __nv_bfloat16*>(q); pp.kq = static_cast<const __nv_bfloat16*>(kq);
  pp.q_rot = q_rot; pp.kq_rot = kq_rot; pp.ctx_off = reinterpret_cast<const long long*>(ctx_off);
  pp.sched = sched; pp.ctx_cap = ctx_cap;
  pp.B = B; pp.k = k; pp.P = P; pp.Tq = Tq; pp.Hq = Hq; pp.Hkv = Hkv; pp.nl = nl; pp.n_gangs = n_gangs;
  pp.To = To; pp.nshots_dev = extra.nshots_dev; pp.status = status;
  if (extra.pass.theta != nullptr) memcpy(pp.theta, extra.pass.theta, D / 2 * sizeof(double));
  else ads_rope_theta(model->rope_base, D, pp.theta);
  for (int i = 0; i < kMaxProbes; ++i) pp.nshots[i] = i < P ? probe_nshots[i] : 0;
  const long long n_tok = (long long)B * nl * P * To;
  const long long n_groups = (n_tok * kPrepParts + 7) / 8;
  pp.tok_blocks = (int)(n_groups < 3 * n_sm ? n_groups : 3 * n_sm);       // what is resident at a time
  ads_launch_dependent(attn_prep_kernel<D>, (unsigned)(1 + pp.ent.blocks + pp.map_blocks + pp.tok_blocks), 256, 0, st, pp);
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;

  // ---- main kernel
  AttnParams ap = {};
  ap.sched = sched; ap.o_part = o_part; ap.ml_part = ml_part;
  ap.out = static_cast<__nv_bfloat16*>(out); ap.lse = lse; ap.status = status;
  ap.B = B; ap.P = P; ap.Tq = Tq; ap.Hq = Hq; ap.Hkv = Hkv; ap.G = G; ap.nl = nl; ap.To = To;
  ap.g_magic = ((1ull << 32) + G - 1) / G;
  ap.n_mt = pl.n_mt; ap.n_mp = pl.n_mp; ap.gang = pl.gang; ap.n_gangs = n_gangs;
  const float scale = model->softmax_scale > 0.f ? model->softmax_scale : 1.0f / sqrtf((float)D);
  ap.scale_log2 = scale * 1.4426950408889634f;
  // the same request for D = 64 as for D = 128: one CTA per SM in every variant
  const int smem = mode == kModeVPool ? (int)AttnSmem<128, kModeVPool>::kTotal
                   : mode == kModeFused ? (int)AttnSmem<128, kModeFused>::kTotal : (int)AttnSmem<128, kModeCache>::kTotal;
  static bool attr_done[3][kAdsMaxDevices] = {{false}, {false}, {false}};   // per template instance (D, mode) and device
  if (g_profile) ADS_CHECK_CUDA(cudaEventRecord(g_profile_ev[0], st));
  if (mode == kModeCache) {
    if (ads_set_max_smem(attn_main_kernel<D, kModeCache>, smem, attr_done[0]) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
    ads_launch_dependent(attn_main_kernel<D, kModeCache>, (unsigned)(n_gangs * pl.gang), kAttnThreads, smem, st,
        tm_q, tm_kctx, tm_vctx, tm_kown, tm_vown, vmaps, kmaps, ap);
  } else {
    ap.row_map = row_map; ap.off_map = off_map; ap.k_pos_mode = model->k_pos_mode;
    ap.ctx_cap = ctx_cap; ap.layer_begin = fused->layer_begin;
    for (int i = 0; i < D / 2; ++i) ap.theta[i] = pp.theta[i];
    if (mode == kModeFused) {
      if (ads_set_max_smem(attn_main_kernel<D, kModeFused>, smem, attr_done[1]) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
      ads_launch_dependent(attn_main_kernel<D, kModeFused>, (unsigned)(n_gangs * pl.gang), kFusedThreads, smem, st,
          tm_q, tm_kctx, tm_vctx, tm_kown, tm_vown, vmaps, kmaps, ap);
    } else {
      if (ads_set_max_smem(attn_main_kernel<D, kModeVPool>, smem, attr_done[2]) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
      ads_launch_dependent(attn_main_kernel<D, kModeVPool>, (unsigned)(n_gangs * pl.gang), kAttnThreads, smem, st,
          tm_q, tm_kctx, tm_vctx, tm_kown, tm_vown, vmaps, kmaps, ap);
    }
  }
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  if (g_profile) {
    ADS_CHECK_CUDA(cudaEventRecord(g_profile_ev[1], st));
    g_profile_valid = true;
  }

  // ---- merge the units that a range boundary cut
  CombineParams cp;
  cp.sched = sched; cp.o_part = o_part; cp.ml_part = ml_part;
  cp.out = ap.out; cp.lse = lse;
  cp.Tq = Tq; cp.Hq = Hq; cp.G = G; cp.n_mp = pl.n_mp;
  // (at most one cut unit per range, and no more than there are units: a small call would launch mostly empty blocks)
  const long long units = (long long)B * P * nl * Hkv;
  cp.units = (int)(units < n_gangs ? units : n_gangs);
  cp.ent = pp.ent;
  dim3 grid((unsigned)cp.units, (unsigned)((Tq * G + 8 * kCombineRows - 1) / (8 * kCombineRows)), D / (16 * kCombineSteps));
  if (cp.ent.blocks > 0) {             // as many more columns of the grid as hold a block for every query
    const unsigned column = grid.y * grid.z;
    grid.x += ((unsigned)(cp.ent.R / cp.ent.rows_per_group) + column - 1) / column;
  }
  ads_launch_dependent(attn_combine_kernel<D>, grid, 256, 0, st, cp);
  return ads_launch_status();
}

}  // namespace

extern "C" size_t adapshot_attn_workspace_bytes(const adapshot_model_t* model, int32_t B, int32_t P,
                                                int32_t Tq, int32_t n_layers_in_call, int64_t ctx_cap) {
  if (model == nullptr || !attn_shape_ok(model) || B <= 0 || P <= 0 || Tq <= 0 || n_layers_in_call <= 0 ||
      ctx_cap <= 0)
    return 0;
  return make_plan(model, B, P, Tq, n_layers_in_call).total;
}

int ads_query_attn(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx, int64_t ctx_cap,
                   const int64_t* ctx_off, int32_t B, int32_t k, const int32_t* probe_nshots, int32_t P, const void* q,
                   const void* kq, const void* vq, int32_t Tq, int32_t layer_begin, int32_t layer_end, void* out,
                   float* lse, uint32_t flags, void* ws, size_t ws_bytes, int32_t* status, void* stream,
                   const AdsPass* pass) {
  if (model == nullptr || k_ctx == nullptr || v_ctx == nullptr || ctx_off == nullptr || probe_nshots == nullptr ||
      q == nullptr || kq == nullptr || vq == nullptr || out == nullptr || ws == nullptr)
    return ADAPSHOT_EINVAL;
  if (B <= 0 || k <= 0 || Tq <= 0 || ctx_cap <= 0 || flags != 0) return ADAPSHOT_EINVAL;
  if (model->dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (!attn_shape_ok(model)) return ADAPSHOT_ESHAPE;
  if (layer_begin < 0 || layer_end <= layer_begin || layer_end > model->n_layers) return ADAPSHOT_ESHAPE;
  if (P < 1 || P > kMaxProbes || (long long)P * B > kMaxPairs) return ADAPSHOT_ESHAPE;
  for (int i = 0; i < P; ++i) {
    if (probe_nshots[i] < 1 || probe_nshots[i] > k) return ADAPSHOT_ESHAPE;
    if (i > 0 && probe_nshots[i] <= probe_nshots[i - 1]) return ADAPSHOT_ESHAPE;
  }
  if (!ads_aligned16(k_ctx) || !ads_aligned16(v_ctx) || !ads_aligned16(q) || !ads_aligned16(kq) ||
      !ads_aligned16(vq) || !ads_aligned16(out) || ((uintptr_t)ws & 255u))
    return ADAPSHOT_EALIGN;
  if (ctx_cap > (1ll << 31) - 256) return ADAPSHOT_ESHAPE;
  const int nl = layer_end - layer_begin;
  const AttnPlan pl = make_plan(model, B, P, Tq, nl);
  if (ws_bytes < pl.total) return ADAPSHOT_ECAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  AttnExtra extra;
  if (pass != nullptr) extra.pass = *pass;
  if (model->head_dim == 128)
    return launch_attn<128>(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, nl, out,
                            lse, pl, ws, status, st, nullptr, kModeCache, extra);
  return launch_attn<64>(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, nl, out,
                         lse, pl, ws, status, st, nullptr, kModeCache, extra);
}

extern "C" int adapshot_query_attn(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx, int64_t ctx_cap,
                                   const int64_t* ctx_off, int32_t B, int32_t k, const int32_t* probe_nshots, int32_t P,
                                   const void* q, const void* kq, const void* vq, int32_t Tq, int32_t layer_begin,
                                   int32_t layer_end, void* out, float* lse, uint32_t flags, void* ws, size_t ws_bytes,
                                   int32_t* status, void* stream) {
  return ads_query_attn(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, layer_begin,
                        layer_end, out, lse, flags, ws, ws_bytes, status, stream, nullptr);
}

extern "C" size_t adapshot_attn_fused_workspace_bytes(const adapshot_model_t* model, int32_t B, int32_t P,
                                                      int32_t Tq, int32_t n_layers_in_call, int64_t ctx_cap) {
  if (model == nullptr || !attn_shape_ok(model) || B <= 0 || P <= 0 || Tq <= 0 || n_layers_in_call <= 0 ||
      ctx_cap <= 0)
    return 0;
  return make_plan(model, B, P, Tq, n_layers_in_call, ctx_cap).total;
}

int ads_query_attn_fused(const adapshot_model_t* model, const adapshot_pool_t* pool, const int32_t* sel_idx,
                         const int64_t* ctx_off, int64_t ctx_cap, int32_t B, int32_t k, const int32_t* probe_nshots,
                         int32_t P, const void* q, const void* kq, const void* vq, int32_t Tq, int32_t layer_begin,
                         int32_t layer_end, void* out, float* lse, uint32_t flags, void* ws, size_t ws_bytes,
                         int32_t* status, void* stream, const AdsPass* pass) {
  if (model == nullptr || pool == nullptr || sel_idx == nullptr || ctx_off == nullptr || probe_nshots == nullptr ||
      q == nullptr || kq == nullptr || vq == nullptr || out == nullptr || ws == nullptr)
    return ADAPSHOT_EINVAL;
  if (pool->k == nullptr || pool->v == nullptr || pool->shot_off == nullptr || pool->n_shots <= 0 ||
      pool->pool_tokens <= 0)
    return ADAPSHOT_EINVAL;
  if (B <= 0 || k <= 0 || Tq <= 0 || ctx_cap <= 0 || flags != 0) return ADAPSHOT_EINVAL;
  if (model->dtype != ADAPSHOT_BF16 || (model->k_pos_mode != 0 && model->k_pos_mode != 1)) return ADAPSHOT_EUNSUPPORTED;
  if (!attn_shape_ok(model)) return ADAPSHOT_ESHAPE;
  if (!(model->rope_base > 1.0)) return ADAPSHOT_EINVAL;
  if (layer_begin < 0 || layer_end <= layer_begin || layer_end > model->n_layers) return ADAPSHOT_ESHAPE;
  if (P < 1 || P > kMaxProbes || (long long)P * B > kMaxPairs || k > pool->n_shots) return ADAPSHOT_ESHAPE;
  for (int i = 0; i < P; ++i) {
    if (probe_nshots[i] < 1 || probe_nshots[i] > k) return ADAPSHOT_ESHAPE;
    if (i > 0 && probe_nshots[i] <= probe_nshots[i - 1]) return ADAPSHOT_ESHAPE;
  }
  if (!ads_aligned16(pool->k) || !ads_aligned16(pool->v) || !ads_aligned16(q) || !ads_aligned16(kq) ||
      !ads_aligned16(vq) || !ads_aligned16(out) || ((uintptr_t)ws & 255u) || ((uintptr_t)sel_idx & 3u))
    return ADAPSHOT_EALIGN;
  if (ctx_cap > (1ll << 31) - 256 || pool->pool_tokens > (1ll << 31) - 1) return ADAPSHOT_ESHAPE;
  const int nl = layer_end - layer_begin;
  const AttnPlan pl = make_plan(model, B, P, Tq, nl, ctx_cap);
  if (ws_bytes < pl.total) return ADAPSHOT_ECAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  AttnExtra extra;
  if (pass != nullptr) extra.pass = *pass;
  FusedSrc src;
  src.pool = pool; src.sel_idx = sel_idx; src.layer_begin = layer_begin;
  if (model->head_dim == 128)
    return launch_attn<128>(model, nullptr, nullptr, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, nl,
                            out, lse, pl, ws, status, st, &src, kModeFused, extra);
  return launch_attn<64>(model, nullptr, nullptr, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, nl, out,
                         lse, pl, ws, status, st, &src, kModeFused, extra);
}

extern "C" int adapshot_query_attn_fused(const adapshot_model_t* model, const adapshot_pool_t* pool,
                                         const int32_t* sel_idx, const int64_t* ctx_off, int64_t ctx_cap, int32_t B,
                                         int32_t k, const int32_t* probe_nshots, int32_t P, const void* q,
                                         const void* kq, const void* vq, int32_t Tq, int32_t layer_begin,
                                         int32_t layer_end, void* out, float* lse, uint32_t flags, void* ws,
                                         size_t ws_bytes, int32_t* status, void* stream) {
  return ads_query_attn_fused(model, pool, sel_idx, ctx_off, ctx_cap, B, k, probe_nshots, P, q, kq, vq, Tq, layer_begin,
                              layer_end, out, lse, flags, ws, ws_bytes, status, stream, nullptr);
}

extern "C" size_t adapshot_attn_vpool_workspace_bytes(const adapshot_model_t* model, int32_t B, int32_t P,
                                                      int32_t Tq, int32_t n_layers_in_call, int64_t ctx_cap) {
  if (model == nullptr || !attn_shape_ok(model) || B <= 0 || P <= 0 || Tq <= 0 || n_layers_in_call <= 0 ||
      ctx_cap <= 0)
    return 0;
  return make_plan(model, B, P, Tq, n_layers_in_call, ctx_cap).total;
}

int ads_query_attn_vpool(const adapshot_model_t* model, const adapshot_pool_t* pool, const int32_t* sel_idx,
                         const void* k_ctx, int64_t ctx_cap, const int64_t* ctx_off, int32_t B, int32_t k,
                         const int32_t* probe_nshots, int32_t P, const void* q, const void* kq, const void* vq,
                         int32_t Tq, int32_t layer_begin, int32_t layer_end, void* out, float* lse, uint32_t flags,
                         void* ws, size_t ws_bytes, int32_t* status, void* stream, const AdsPass* pass) {
  if (model == nullptr || pool == nullptr || sel_idx == nullptr || k_ctx == nullptr || ctx_off == nullptr ||
      probe_nshots == nullptr || q == nullptr || kq == nullptr || vq == nullptr || out == nullptr || ws == nullptr)
    return ADAPSHOT_EINVAL;
  if (pool->v == nullptr || pool->shot_off == nullptr || pool->n_shots <= 0 || pool->pool_tokens <= 0)
    return ADAPSHOT_EINVAL;
  if (B <= 0 || k <= 0 || Tq <= 0 || ctx_cap <= 0 || flags != 0) return ADAPSHOT_EINVAL;
  if (model->dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (!attn_shape_ok(model)) return ADAPSHOT_ESHAPE;
  if (layer_begin < 0 || layer_end <= layer_begin || layer_end > model->n_layers) return ADAPSHOT_ESHAPE;
  if (P < 1 || P > kMaxProbes || (long long)P * B > kMaxPairs || k > pool->n_shots) return ADAPSHOT_ESHAPE;
  for (int i = 0; i < P; ++i) {
    if (probe_nshots[i] < 1 || probe_nshots[i] > k) return ADAPSHOT_ESHAPE;
    if (i > 0 && probe_nshots[i] <= probe_nshots[i - 1]) return ADAPSHOT_ESHAPE;
  }
  if (!ads_aligned16(pool->v) || !ads_aligned16(k_ctx) || !ads_aligned16(q) || !ads_aligned16(kq) ||
      !ads_aligned16(vq) || !ads_aligned16(out) || ((uintptr_t)ws & 255u) || ((uintptr_t)sel_idx & 3u))
    return ADAPSHOT_EALIGN;
  if (ctx_cap > (1ll << 31) - 256 || pool->pool_tokens > (1ll << 31) - 1) return ADAPSHOT_ESHAPE;
  const int nl = layer_end - layer_begin;
  const AttnPlan pl = make_plan(model, B, P, Tq, nl, ctx_cap);
  if (ws_bytes < pl.total) return ADAPSHOT_ECAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  AttnExtra extra;
  if (pass != nullptr) extra.pass = *pass;
  FusedSrc src;
  src.pool = pool; src.sel_idx = sel_idx; src.layer_begin = layer_begin;
  if (model->head_dim == 128)
    return launch_attn<128>(model, k_ctx, nullptr, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, nl, out,
                            lse, pl, ws, status, st, &src, kModeVPool, extra);
  return launch_attn<64>(model, k_ctx, nullptr, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq, nl, out, lse,
                         pl, ws, status, st, &src, kModeVPool, extra);
}

extern "C" int adapshot_query_attn_vpool(const adapshot_model_t* model, const adapshot_pool_t* pool,
                                         const int32_t* sel_idx, const void* k_ctx, int64_t ctx_cap,
                                         const int64_t* ctx_off, int32_t B, int32_t k, const int32_t* probe_nshots,
                                         int32_t P, const void* q, const void* kq, const void* vq, int32_t Tq,
                                         int32_t layer_begin, int32_t layer_end, void* out, float* lse, uint32_t flags,
                                         void* ws, size_t ws_bytes, int32_t* status, void* stream) {
  return ads_query_attn_vpool(model, pool, sel_idx, k_ctx, ctx_cap, ctx_off, B, k, probe_nshots, P, q, kq, vq, Tq,
                              layer_begin, layer_end, out, lse, flags, ws, ws_bytes, status, stream, nullptr);
}

// ---------------------------------------------------------------- literal tree layout
namespace {
// Position ids of the probe tokens of the interleaved sequence: token t of probe j of query b sits
// at L_j + t (the shots keep the positions 0 .. L-1 of their plain concatenation).
struct TreePosArgs { int n[kMaxProbes]; };
__global__ void tree_positions_kernel(const long long* __restrict__ ctx_off, int B, int k, int P, int Tq,
                                           const TreePosArgs a, long long* __restrict__ pos) {
  ads_dependency_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)B * P * Tq) return;
  const int t = (int)(i % Tq), j = (int)((i / Tq) % P), b = (int)(i / ((long long)Tq * P));
  pos[i] = ctx_off[(long long)b * (k + 1) + a.n[j]] + t;
}
}  // namespace

extern "C" int adapshot_tree_layout(const int32_t* seg_kind, const int32_t* seg_len, int32_t n_seg, int32_t k,
                                    int32_t* probe_nshots, int32_t* P_out, int32_t* Tq_out) {
  if (seg_kind == nullptr || seg_len == nullptr || probe_nshots == nullptr || P_out == nullptr || Tq_out == nullptr ||
      n_seg <= 0)
    return ADAPSHOT_EINVAL;
  int shots = 0, P = 0, Tq = 0;
  bool shots_since_probe = false;
  for (int i = 0; i < n_seg; ++i) {
    if (seg_len[i] <= 0) return ADAPSHOT_ESHAPE;
    if (seg_kind[i] == ADAPSHOT_SEG_SHOTS) {
      shots += seg_len[i];
      if (shots > k) return ADAPSHOT_ESHAPE;
      shots_since_probe = true;
    } else if (seg_kind[i] == ADAPSHOT_SEG_PROBE) {
      // every probe follows at least one new shot (nested counts are strictly ascending) and all
      // probes have the same number of tokens
      if (!shots_since_probe || P >= kMaxProbes) return ADAPSHOT_ESHAPE;
      if (P == 0) Tq = seg_len[i];
      else if (seg_len[i] != Tq) return ADAPSHOT_ESHAPE;
      probe_nshots[P++] = shots;
      shots_since_probe = false;
    } else {
      return ADAPSHOT_EINVAL;
    }
  }
  if (P == 0 || shots_since_probe) return ADAPSHOT_ESHAPE;      // the sequence ends with a probe
  *P_out = P;
  *Tq_out = Tq;
  return ADAPSHOT_OK;
}

extern "C" int adapshot_tree_attn(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx,
                                  int64_t ctx_cap, const int64_t* ctx_off, int32_t B, int32_t k,
                                  const int32_t* seg_kind, const int32_t* seg_len, int32_t n_seg,
                                  const void* q_seq, const void* kq_seq, const void* vq_seq,
                                  int32_t layer_begin, int32_t layer_end, void* out_seq, float* lse,
                                  int64_t* pos_seq, uint32_t flags, void* ws, size_t ws_bytes, int32_t* status,
                                  void* stream) {
  int32_t nshots[kMaxProbes], P = 0, Tq = 0;
  if (model == nullptr || ctx_off == nullptr) return ADAPSHOT_EINVAL;
  const int rc = adapshot_tree_layout(seg_kind, seg_len, n_seg, k, nshots, &P, &Tq);
  if (rc != ADAPSHOT_OK) return rc;
  // the probe tokens of the sequence, in sequence order, are [P][T_q]: the per-probe call's layout
  const int rc2 = adapshot_query_attn(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, nshots, P, q_seq, kq_seq, vq_seq,
                                      Tq, layer_begin, layer_end, out_seq, lse, flags, ws, ws_bytes, status, stream);
  if (rc2 != ADAPSHOT_OK || pos_seq == nullptr) return rc2;
  if ((uintptr_t)pos_seq & 7u) return ADAPSHOT_EALIGN;
  TreePosArgs a;
  for (int i = 0; i < kMaxProbes; ++i) a.n[i] = i < P ? nshots[i] : 0;
  const long long n = (long long)B * P * Tq;
  ads_launch_dependent(tree_positions_kernel, (unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream),
      reinterpret_cast<const long long*>(ctx_off), B, k, P, Tq, a, reinterpret_cast<long long*>(pos_seq));
  return ads_launch_status();
}

// ------------------------------------------------------------------------ decode step
extern "C" size_t adapshot_decode_workspace_bytes(const adapshot_model_t* model, int32_t B, int32_t T_new,
                                                  int32_t T_own, int32_t n_layers_in_call) {
  if (model == nullptr || !attn_shape_ok(model) || B <= 0 || T_new <= 0 || T_own < T_new || n_layers_in_call <= 0)
    return 0;
  const size_t rows = ads_decode_rows_workspace(model, B), plan = make_plan(model, B, 1, T_new, n_layers_in_call, 0, T_own).total;
  if (!ads_decode_rows_fit(model, T_new)) return plan;
  // (a larger context only ever speaks for the kernel that streams)
  return ads_decode_rows_pay(model, B, T_new, T_own, 1) || rows > plan ? rows : plan;
}

extern "C" int adapshot_decode_attn(const adapshot_model_t* model, const void* k_ctx, const void* v_ctx,
                                    int64_t ctx_cap, const int64_t* ctx_off, int32_t B, int32_t k,
                                    const int32_t* n_shots, const void* q_new, const void* k_own,
                                    const void* v_own, int32_t T_new, int32_t T_own, int32_t layer_begin,
                                    int32_t layer_end, void* out, float* lse, uint32_t flags, void* ws,
                                    size_t ws_bytes, int32_t* status, void* stream) {
  if (model == nullptr || k_ctx == nullptr || v_ctx == nullptr || ctx_off == nullptr || n_shots == nullptr ||
      q_new == nullptr || k_own == nullptr || v_own == nullptr || out == nullptr || ws == nullptr)
    return ADAPSHOT_EINVAL;
  if (B <= 0 || k <= 0 || T_new <= 0 || ctx_cap <= 0 || flags != 0) return ADAPSHOT_EINVAL;
  if (T_own < T_new) return ADAPSHOT_ESHAPE;
  if (model->dtype != ADAPSHOT_BF16) return ADAPSHOT_EUNSUPPORTED;
  if (!attn_shape_ok(model)) return ADAPSHOT_ESHAPE;
  if (layer_begin < 0 || layer_end <= layer_begin || layer_end > model->n_layers) return ADAPSHOT_ESHAPE;
  if (B > kMaxPairs) return ADAPSHOT_ESHAPE;
  if (!ads_aligned16(k_ctx) || !ads_aligned16(v_ctx) || !ads_aligned16(q_new) || !ads_aligned16(k_own) ||
      !ads_aligned16(v_own) || !ads_aligned16(out) || ((uintptr_t)ws & 255u) || ((uintptr_t)n_shots & 3u))
    return ADAPSHOT_EALIGN;
  if (ctx_cap > (1ll << 31) - 256) return ADAPSHOT_ESHAPE;
  const int nl = layer_end - layer_begin;
  // Up to 32 rows per KV head: the kernel that streams K/V through warp-level tiles (decode.cu) where it pays: 256 against
  // 376 us at 4 rows and 32 requests.  The line is where its accumulators stop fitting two CTAs per SM; more rows
  // fill the 128-row tiles of the prefill kernels better as well.  A workspace that only it can do with is taken, too.
  if (ads_decode_rows_fit(model, T_new) &&
      (ads_decode_rows_pay(model, B, T_new, T_own, ctx_cap) || ws_bytes < make_plan(model, B, 1, T_new, nl, 0, T_own).total)) {
    if (ws_bytes < ads_decode_rows_workspace(model, B)) return ADAPSHOT_ECAPACITY;
    return ads_decode_rows(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, n_shots, q_new, k_own, v_own, T_new, T_own, nl,
                           out, lse, ws, status, static_cast<cudaStream_t>(stream));
  }
  const AttnPlan pl = make_plan(model, B, 1, T_new, nl, 0, T_own);
  if (ws_bytes < pl.total) return ADAPSHOT_ECAPACITY;
  AttnExtra extra;
  extra.To = T_own;
  extra.nshots_dev = n_shots;
  const int32_t one = 1;      // (placeholder for the host list: the per-query device counts are used)
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (model->head_dim == 128)
    return launch_attn<128>(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, &one, 1, q_new, k_own, v_own, T_new, nl, out,
                            lse, pl, ws, status, st, nullptr, kModeCache, extra);
  return launch_attn<64>(model, k_ctx, v_ctx, ctx_cap, ctx_off, B, k, &one, 1, q_new, k_own, v_own, T_new, nl, out,
                         lse, pl, ws, status, st, nullptr, kModeCache, extra);
}

extern "C" int adapshot_profile(int enable) {
  if (enable && g_profile_ev[0] == nullptr) {
    ADS_CHECK_CUDA(cudaEventCreate(&g_profile_ev[0]));
    ADS_CHECK_CUDA(cudaEventCreate(&g_profile_ev[1]));
  }
  g_profile = enable != 0;
  g_profile_valid = false;
  return ADAPSHOT_OK;
}

extern "C" float adapshot_profile_attn_main_ms(void) {
  if (!g_profile_valid) return -1.f;
  float ms = -1.f;
  if (cudaEventSynchronize(g_profile_ev[1]) != cudaSuccess) return -1.f;
  if (cudaEventElapsedTime(&ms, g_profile_ev[0], g_profile_ev[1]) != cudaSuccess) return -1.f;
  return ms;
}

extern "C" int adapshot_selftest_wait_timeout(int32_t* status, long long* cycles, void* stream) {
  if (status == nullptr || cycles == nullptr) return ADAPSHOT_EINVAL;
  wait_timeout_selftest_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(status, cycles);
  return ads_launch_status();
}
