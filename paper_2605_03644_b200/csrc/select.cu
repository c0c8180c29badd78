// Semantic shot selection (paper Sec. 4.1 ranking, Sec. 4.2 "rank in descending
// order and select the top k"): cosine of the query embedding against every cached
// shot embedding, then the top k with ties broken by the lower shot id.
//
// The ranking must equal that of an fp64 evaluation of the same formula, so the
// fp32 products (exact in fp64) are accumulated in fp64 and scores are compared in
// fp64, as 64-bit sort keys.  Batches of queries go through fp64 matrix instructions, one or two
// queries through a warp per shot; the top k are found by rank counting for small pools
// and by a radix selection in front of a sort of the few candidates otherwise.
#include "common.cuh"

namespace {

constexpr int kSortCap = 8192;      // candidates one CTA sorts in shared memory

__device__ __forceinline__ unsigned long long desc_key(double s) { return ads_desc_key(s); }
__device__ __forceinline__ double key_score(unsigned long long k) { return ads_key_score(k); }

// sort key of cos = <q, e> / (|q| |e|), 0 where either norm is 0
__device__ __forceinline__ unsigned long long cosine_key(double dot, double qq, double nn) {
  const double den = sqrt(qq) * sqrt(nn);
  return desc_key(den > 0.0 ? dot / den : 0.0);
}

// One warp per pool row i, for one or two queries: keys[b][i] = sort key of cos(q_b, e_i).
// NV > 0: E = 128 NV, the row is widened to fp64 once and kept in registers for all queries
// (the fp32 -> fp64 conversions are what a row-times-query pass pays for); NV = 0: any E and any B.
template <int NV>
__global__ void __launch_bounds__(256)
cosine_keys_kernel(const float* __restrict__ emb, const float* __restrict__ q_emb, int N, int E,
                   int B, unsigned long long* __restrict__ keys) {
  ads_dependency_wait();
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= N) return;
  const float* e = emb + (long long)row * E;
  double nn = 0.0;
  if constexpr (NV > 0) {
    double ev[4 * NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(e + lane * 4 + 128 * i);
      ev[4 * i] = v.x; ev[4 * i + 1] = v.y; ev[4 * i + 2] = v.z; ev[4 * i + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < 4 * NV; ++j) nn += ev[j] * ev[j];
    nn = warp_sum(nn);
    for (int b = 0; b < B; ++b) {
      const float* q = q_emb + (long long)b * E;
      double acc = 0.0, qq = 0.0;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(q + lane * 4 + 128 * i));
        const double w0 = w.x, w1 = w.y, w2 = w.z, w3 = w.w;
        acc += ev[4 * i] * w0 + ev[4 * i + 1] * w1 + ev[4 * i + 2] * w2 + ev[4 * i + 3] * w3;
        qq += w0 * w0 + w1 * w1 + w2 * w2 + w3 * w3;
      }
      acc = warp_sum(acc);
      qq = warp_sum(qq);
      if (lane == 0) keys[(long long)b * N + row] = cosine_key(acc, qq, nn);
    }
    return;
  }
  const bool vec_ok = (E & 3) == 0;
  if (vec_ok) {
    for (int i = lane * 4; i < E; i += 128) {
      float4 v = *reinterpret_cast<const float4*>(e + i);
      nn += (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z + (double)v.w * v.w;
    }
  } else {
    for (int i = lane; i < E; i += 32) nn += (double)e[i] * e[i];
  }
  nn = warp_sum(nn);
  for (int b = 0; b < B; ++b) {
    const float* q = q_emb + (long long)b * E;
    double acc = 0.0, qq = 0.0;
    if (vec_ok) {
      for (int i = lane * 4; i < E; i += 128) {
        float4 v = *reinterpret_cast<const float4*>(e + i);   // L1-resident after the first pass
        float4 w = __ldg(reinterpret_cast<const float4*>(q + i));
        acc += (double)v.x * w.x + (double)v.y * w.y + (double)v.z * w.z + (double)v.w * w.w;
        qq += (double)w.x * w.x + (double)w.y * w.y + (double)w.z * w.z + (double)w.w * w.w;
      }
    } else {
      for (int i = lane; i < E; i += 32) {
        acc += (double)e[i] * q[i];
        qq += (double)q[i] * q[i];
      }
    }
    acc = warp_sum(acc);
    qq = warp_sum(qq);
    if (lane == 0) keys[(long long)b * N + row] = cosine_key(acc, qq, nn);
  }
}

// c (16 x 8) += a (16 x 8) b (8 x 8), fp64
__device__ __forceinline__ void mma_f64(double (&c)[4], const double (&a)[4], const double (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
               : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b[0]), "d"(b[1]));
}

// The same for batches: a CTA takes 16 RB shots and 8 NB queries, its eight warps share the embedding's length
// and are summed in a fixed order through shared memory.  Bound by the fp64 units; the operands come straight
// from memory as fp32 (a lane's four consecutive elements are the k slots lane % 4 and lane % 4 + 4 of two
// instructions), so an element is widened once per 8 NB queries or 16 RB shots instead of once per product, which is
// what the warp-per-shot form above spends its time on.  Norms are summed from the same registers.  E % 16 == 0.
// (20000 shots x 768, 16 queries: 140 -> 24 us; 8192 x 1024, 32 queries: 115 -> 25 us.)
constexpr int kMmaWarps = 8;
template <int NB, int RB>
__global__ void __launch_bounds__(32 * kMmaWarps, RB == 2 ? 2 : 3)
cosine_mma_kernel(const float* __restrict__ emb, const float* __restrict__ q_emb, int N, int E, int B,
                  unsigned long long* __restrict__ keys) {
  __shared__ double dot_s[kMmaWarps][8 * NB][16 * RB + 1];
  __shared__ double nn_s[kMmaWarps][16 * RB], qq_s[kMmaWarps][8 * NB];
  ads_dependency_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int row0 = blockIdx.x * 16 * RB, q0 = blockIdx.y * 8 * NB;
  const int steps = E / 16, s0 = warp * steps / kMmaWarps, s1 = (warp + 1) * steps / kMmaWarps;
  const float4* ap[2 * RB];
  const float4* bp[NB];
#pragma unroll
  for (int r = 0; r < 2 * RB; ++r)
    ap[r] = reinterpret_cast<const float4*>(emb + (long long)min(row0 + 8 * r + g, N - 1) * E) + s0 * 4 + t;
#pragma unroll
  for (int n = 0; n < NB; ++n)
    bp[n] = reinterpret_cast<const float4*>(q_emb + (long long)min(q0 + 8 * n + g, B - 1) * E) + s0 * 4 + t;
  double c[RB][NB][4] = {}, nn[2 * RB] = {}, qq[NB] = {};
  float4 av[2 * RB], bv[NB];
  auto load = [&]() {
#pragma unroll
    for (int r = 0; r < 2 * RB; ++r) { av[r] = __ldg(ap[r]); ap[r] += 4; }
#pragma unroll
    for (int n = 0; n < NB; ++n) { bv[n] = __ldg(bp[n]); bp[n] += 4; }
  };
  if (s0 < s1) load();
  for (int s = s0; s < s1; ++s) {
    double a[2 * RB][4], b[NB][4];
#pragma unroll
    for (int r = 0; r < 2 * RB; ++r) { a[r][0] = av[r].x; a[r][1] = av[r].y; a[r][2] = av[r].z; a[r][3] = av[r].w; }
#pragma unroll
    for (int n = 0; n < NB; ++n) { b[n][0] = bv[n].x; b[n][1] = bv[n].y; b[n][2] = bv[n].z; b[n][3] = bv[n].w; }
    if (s + 1 < s1) load();
#pragma unroll
    for (int r = 0; r < 2 * RB; ++r)
#pragma unroll
      for (int e = 0; e < 4; ++e) nn[r] += a[r][e] * a[r][e];
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) qq[n] += b[n][e] * b[n][e];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int m = 0; m < RB; ++m)
#pragma unroll
        for (int n = 0; n < NB; ++n) {
          const double aa[4] = {a[2 * m][2 * h], a[2 * m + 1][2 * h], a[2 * m][2 * h + 1], a[2 * m + 1][2 * h + 1]};
          const double bb[2] = {b[n][2 * h], b[n][2 * h + 1]};
          mma_f64(c[m][n], aa, bb);
        }
  }
#pragma unroll
  for (int m = 0; m < RB; ++m)
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) dot_s[warp][8 * n + 2 * t + (e & 1)][16 * m + 8 * (e >> 1) + g] = c[m][n][e];
#pragma unroll
  for (int r = 0; r < 2 * RB; ++r) {
    nn[r] += __shfl_xor_sync(0xffffffffu, nn[r], 1);
    nn[r] += __shfl_xor_sync(0xffffffffu, nn[r], 2);
    if (t == 0) nn_s[warp][8 * r + g] = nn[r];
  }
#pragma unroll
  for (int n = 0; n < NB; ++n) {
    qq[n] += __shfl_xor_sync(0xffffffffu, qq[n], 1);
    qq[n] += __shfl_xor_sync(0xffffffffu, qq[n], 2);
    if (t == 0) qq_s[warp][8 * n + g] = qq[n];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 16 * RB * 8 * NB; i += 32 * kMmaWarps) {
    const int r = i % (16 * RB), q = i / (16 * RB);
    if (row0 + r >= N || q0 + q >= B) continue;
    double d = 0.0, n2 = 0.0, q2 = 0.0;
#pragma unroll
    for (int w = 0; w < kMmaWarps; ++w) {
      d += dot_s[w][q][r];
      n2 += nn_s[w][r];
      q2 += qq_s[w][q];
    }
    keys[(long long)(q0 + q) * N + row0 + r] = cosine_key(d, q2, n2);
  }
}

__device__ __forceinline__ bool pair_less(unsigned long long ka, int ia, unsigned long long kb, int ib) {
  return ka < kb || (ka == kb && ia < ib);
}

// Top k by radix selection, one CTA per query.  The keys' interval is narrowed, 4096 bins at a time, until
// the bin that holds the k-th key and everything in front of it fit the candidate area; up to 1024 candidates are then
// put in order by dealing them out to 4096 bins once more, more of them, or those that crowd a bin, by a bitonic sort.  The first pass bins by the score's
// sign, exponent and five bits more (cosines and attention masses both spread over many of them), the following ones
// divide the bin's interval evenly, so two passes nearly always do; equal keys without end are cut by id.  Bound by the
// instructions of one SM per query: a pass reads the keys once (the second one from L1) with eight loads in flight per
// thread.  A cluster of eight CTAs per query that added their histograms up through distributed shared memory was slower
// (40 us against 21 at 20000 keys): the cluster barriers cost more than the counting.  (20000 keys, k = 512, 16 queries: one
// 8192-entry bitonic sort per chunk 159 us, candidates sorted in 55 steps and bins by compares and selects 20.8, now 16.3; 8192
// keys, k = 512, 32 queries 145, 14.6 and 11.2; 4096 keys, k = 256, 8 queries 11.0 and 9.6.)
constexpr int kSelThreads = 1024;
constexpr int kSelBins = 4096;
constexpr int kBinMost = 128;         // candidates in one bin that are ordered by comparing each with all (40 copies of every shot: 21.6 us, 25.2 by sorting)

// First-pass bins, ascending with the key: 0 = scores of 2 and more, 1 .. 2040 = positive scores below that in 32nds
// of an octave (63 octaves), 2041 = smaller ones, then the negative scores in the same way.
constexpr int kBinHi = (1023 + 1) << 5, kBinLo = kBinHi - 2040;
constexpr int kBinShift = 47;                     // leaves the sign, the exponent and 5 bits
__device__ __forceinline__ int first_bin(unsigned long long key) {
  const int v = (int)((uint32_t)(key >> 32) >> (kBinShift - 32));     // 17 bits: those of a positive score count down
  const bool neg = v >= 0x10000;
  const int m = neg ? v - 0x10000 : 0xffff - v;
  const int mid = min(max(m - kBinLo, -1), 2040);
  return neg ? 2043 + mid : 2040 - mid;
}
__device__ __forceinline__ void first_bin_interval(int bin, unsigned long long* lo, unsigned long long* hi) {
  int a, b;                                       // first and last v of the bin
  if (bin == 0) { a = 0; b = 0xffff - kBinHi; }
  else if (bin <= 2040) { a = b = 0xffff - (kBinLo + 2040 - bin); }
  else if (bin == 2041) { a = 0xffff - (kBinLo - 1); b = 0xffff; }
  else if (bin == 2042) { a = 0x10000; b = 0x10000 + kBinLo - 1; }
  else if (bin <= 4082) { a = b = 0x10000 + kBinLo + bin - 2043; }
  else { a = 0x10000 + kBinHi; b = 0x1ffff; }
  *lo = (unsigned long long)a << kBinShift;
  *hi = ((unsigned long long)b << kBinShift) | ((1ull << kBinShift) - 1);
}

// The candidates of a query one of whose bins is crowded, by a bitonic sort, ascending on (key, id), one per thread (padding: the largest
// key and id), exchanged within a warp by shuffles.  (Calls of 16 queries over 8192 shots, all scores equal, k = 512: 25.0 us, 30.5
// where every exchange goes through shared memory as below.  Not inlined: the calls without a crowded bin 13.72 us, 13.95 with it inlined.)
__device__ __noinline__ void sort_candidates(unsigned long long key, int id, int n, int n_out, unsigned long long* ckey, int* cid,
                                             int32_t* idx, float* score) {
  int n_pow2 = 32;
  while (n_pow2 < n) n_pow2 <<= 1;
  const int tid = threadIdx.x;
  if (tid >= n_pow2) return;                        // (whole warps)
  auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(n_pow2) : "memory"); };
  for (int size = 2; size <= n_pow2; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      unsigned long long ko;
      int io;
      if (stride >= 32) {
        sync();
        ckey[tid] = key;
        cid[tid] = id;
        sync();
        ko = ckey[tid ^ stride];
        io = cid[tid ^ stride];
      } else {
        ko = __shfl_xor_sync(0xffffffffu, key, stride);
        io = __shfl_xor_sync(0xffffffffu, id, stride);
      }
      const bool keep_low = ((tid & stride) == 0) == ((tid & size) == 0);
      if (pair_less(ko, io, key, id) == keep_low) {
        key = ko;
        id = io;
      }
    }
  }
  if (tid < n_out) {
    idx[tid] = id;
    if (score != nullptr) score[tid] = (float)key_score(key);
  }
}

__global__ void __launch_bounds__(kSelThreads)
radix_topk_kernel(const unsigned long long* __restrict__ all_keys, int N, int k, int want, int32_t* __restrict__ final_idx,
                  float* __restrict__ final_score) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* ckey = reinterpret_cast<unsigned long long*>(smem_raw);     // [want] candidates
  int* cid = reinterpret_cast<int*>(ckey + want);                                 // [want]
  int* hist = cid + want;                                                         // [kSelBins]
  __shared__ int warp_sum_s[32], bin_s, before_s, inside_s, n_s;
  __shared__ unsigned long long warp_min_s[32], warp_max_s[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const unsigned long long* keys = all_keys + (long long)b * N;
  ads_dependency_wait();
  constexpr int kFly = 8;

  // This thread's four bins and how many entries lie in front of them (a barrier in between: the caller writes before it).
  auto bins_before = [&](int (&h)[4]) -> int {
    const int4 h4 = *reinterpret_cast<const int4*>(hist + 4 * tid);
    h[0] = h4.x; h[1] = h4.y; h[2] = h4.z; h[3] = h4.w;
    const int sum = h[0] + h[1] + h[2] + h[3];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) warp_sum_s[warp] = incl;
    __syncthreads();
    return incl - sum + __reduce_add_sync(0xffffffffu, lane < warp ? warp_sum_s[lane] : 0);
  };
  unsigned long long lo = 0, hi = ~0ull;           // keys below lo: taken; above hi: out
  int before = 0, inside = N;                       // how many are below lo, how many in [lo, hi]
  if (tid == 0) n_s = 0;
  for (int pass = 0; before + inside > want && lo < hi; ++pass) {
    int shift = 64 - __clzll((long long)(hi - lo)) - 12;
    if (shift < 0) shift = 0;
    *reinterpret_cast<int4*>(hist + 4 * tid) = make_int4(0, 0, 0, 0);
    __syncthreads();
    for (int i0 = tid; i0 < N; i0 += kFly * kSelThreads) {
      unsigned long long key[kFly];
#pragma unroll
      for (int u = 0; u < kFly; ++u) key[u] = i0 + u * kSelThreads < N ? keys[i0 + u * kSelThreads] : ~0ull;
      if (pass == 0) {
#pragma unroll
        for (int u = 0; u < kFly; ++u)
          if (i0 + u * kSelThreads < N) atomicAdd(hist + first_bin(key[u]), 1);
      } else {
#pragma unroll
        for (int u = 0; u < kFly; ++u)
          if (i0 + u * kSelThreads < N && key[u] >= lo && key[u] <= hi) atomicAdd(hist + (int)((key[u] - lo) >> shift), 1);
      }
    }
    __syncthreads();
    // the bin that holds rank k - 1
    int h[4];
    int at = before + bins_before(h);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (at < k && at + h[u] >= k) {
        bin_s = 4 * tid + u;
        before_s = at;
        inside_s = h[u];
      }
      at += h[u];
    }
    __syncthreads();
    before = before_s;
    inside = inside_s;
    if (pass == 0) {
      first_bin_interval(bin_s, &lo, &hi);
    } else {
      lo += (unsigned long long)bin_s << shift;
      const unsigned long long top = lo + ((1ull << shift) - 1);
      hi = top < hi ? top : hi;
    }
  }
  __syncthreads();

  // candidates: everything up to hi; of more equal keys than there is room for, the lowest ids
  const bool cut = before + inside > want;          // then lo == hi
  int taken = 0;                                    // equal keys with lower ids (cut only)
  for (int i0 = tid; i0 < N + tid; i0 += kFly * kSelThreads) {      // (whole warps: i0 - tid is the same for all)
    unsigned long long key[kFly];
#pragma unroll
    for (int u = 0; u < kFly; ++u) key[u] = i0 + u * kSelThreads < N ? keys[i0 + u * kSelThreads] : ~0ull;
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const int i = i0 + u * kSelThreads;
      bool take = i < N && key[u] <= hi;
      if (cut) {                                    // in id order: a block-wide count of the equal keys
        const bool eq = i < N && key[u] == hi;
        const unsigned m = __ballot_sync(0xffffffffu, eq);
        __syncthreads();
        if (lane == 0) warp_sum_s[warp] = __popc(m);
        __syncthreads();
        const int v = warp_sum_s[lane];
        const int pos = taken + __reduce_add_sync(0xffffffffu, lane < warp ? v : 0) + __popc(m & ((1u << lane) - 1));
        taken += __reduce_add_sync(0xffffffffu, v);
        if (eq) take = before + pos < k;
      }
      const unsigned m = __ballot_sync(0xffffffffu, take);
      if (m == 0) continue;
      int slot = 0;
      if (lane == 0) slot = atomicAdd(&n_s, __popc(m));
      slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(m & ((1u << lane) - 1));
      if (take) {
        ckey[slot] = key[u];
        cid[slot] = i;
      }
    }
  }
  __syncthreads();
  const int n = n_s;
  if (want <= kSelThreads) {
    // One candidate per thread, dealt out to 4096 bins; its place is what lies in front of its bin and what precedes it there.  The bins
    // are of equal width between the smallest and the largest key, or, where that would leave an octave fewer than 32 of them (scores on
    // both sides of zero; 32 queries of 2048 shots, k = 1000: 24.6 us when they crowded a few bins, 10.7 now), those of the first pass.
    unsigned long long* skey = reinterpret_cast<unsigned long long*>(hist + kSelBins);     // [want], by bin
    int* sid = reinterpret_cast<int*>(skey + want);
    const unsigned long long key = tid < n ? ckey[tid] : ~0ull;
    const int id = tid < n ? cid[tid] : 0x7fffffff;
    unsigned long long least = key, most = tid < n ? key : 0;
    auto across = [&]() {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, least, o), c = __shfl_xor_sync(0xffffffffu, most, o);
        least = a < least ? a : least;
        most = c > most ? c : most;
      }
    };
    across();
    if (lane == 0) { warp_min_s[warp] = least; warp_max_s[warp] = most; }
    *reinterpret_cast<int4*>(hist + 4 * tid) = make_int4(0, 0, 0, 0);
    __syncthreads();
    least = warp_min_s[lane];
    most = warp_max_s[lane];
    across();
    int shift = 64 - __clzll((long long)(most - least)) - 12;
    if (shift < 0) shift = 0;
    int bin = 0, nth = 0;
    if (tid < n) {
      if (shift <= kBinShift) bin = (int)((key - least) >> shift);
      else bin = first_bin(key);
      nth = atomicAdd(hist + bin, 1);
    }
    if (!__syncthreads_or(nth >= kBinMost)) {
      int h[4];
      int at = bins_before(h);
      *reinterpret_cast<int4*>(hist + 4 * tid) = make_int4(at, at + h[0], at + h[0] + h[1], at + h[0] + h[1] + h[2]);
      __syncthreads();
      int first = 0, last = 0;
      if (tid < n) {
        first = hist[bin];
        last = bin + 1 < kSelBins ? hist[bin + 1] : n;
        skey[first + nth] = key;
        sid[first + nth] = id;
      }
      __syncthreads();
      int place = first;
      for (int i = first; i < last; ++i) place += pair_less(skey[i], sid[i], key, id) ? 1 : 0;
      if (tid < n && place < k) {
        final_idx[(long long)b * k + place] = id;
        if (final_score != nullptr) final_score[(long long)b * k + place] = (float)key_score(key);
      }
      return;
    }
    sort_candidates(key, id, n, min(k, n), ckey, cid, final_idx + (long long)b * k,
                    final_score == nullptr ? nullptr : final_score + (long long)b * k);
    return;
  }
  // bitonic sort, ascending on (key, id); ids are unique so the order is total
  int n_pow2 = 32;
  while (n_pow2 < n) n_pow2 <<= 1;
  for (int i = n + tid; i < n_pow2; i += kSelThreads) {
    ckey[i] = ~0ull;
    cid[i] = 0x7fffffff;
  }
  __syncthreads();
  for (int size = 2; size <= n_pow2; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int u = tid; u < (n_pow2 >> 1); u += kSelThreads) {
        const int x = 2 * u - (u & (stride - 1)), y = x + stride;
        const bool up = (x & size) == 0;
        const unsigned long long kx = ckey[x], ky = ckey[y];
        const int ix = cid[x], iy = cid[y];
        if (up ? pair_less(ky, iy, kx, ix) : pair_less(kx, ix, ky, iy)) {
          ckey[x] = ky; ckey[y] = kx;
          cid[x] = iy; cid[y] = ix;
        }
      }
      __syncthreads();
    }
  }
  for (int r = tid; r < min(k, n); r += kSelThreads) {
    final_idx[(long long)b * k + r] = cid[r];
    if (final_score != nullptr) final_score[(long long)b * k + r] = (float)key_score(ckey[r]);
  }
}

// Top-k by counting, for small pools: the rank of shot i in the order
// (score descending, id ascending) is the number of shots that precede it; every shot with
// rank < k writes its id to position rank.  No sort and no serial phases: grid (N / 16, B),
// 16 candidates per CTA, the comparison range split over sixteen groups of 16 threads.
// "key_j precedes key_i" = key_j < key_i, or equal keys and j < i, = key_j < key_i + (j < i).
constexpr int kRankThreads = 256, kRankCand = 16, kRankTile = 2048;
constexpr int kRankParts = kRankThreads / kRankCand;

__global__ void __launch_bounds__(kRankThreads)
rank_topk_kernel(const unsigned long long* __restrict__ all_keys, int N, int k,
                 int32_t* __restrict__ final_idx, float* __restrict__ final_score) {
  __shared__ __align__(16) unsigned long long keys[kRankTile];
  __shared__ int part_cnt[kRankThreads];
  ads_dependency_wait();
  const int b = blockIdx.y;
  const int tid = threadIdx.x;
  const unsigned long long* gkeys = all_keys + (long long)b * N;
  auto key_of = [&](int j) -> unsigned long long { return gkeys[j]; };
  const int i = blockIdx.x * kRankCand + (tid & (kRankCand - 1));
  const int part = tid / kRankCand;                       // which part of every tile this thread scans
  const unsigned long long ki = i < N ? key_of(i) : ~0ull;
  const unsigned long long ki_le = ki == ~0ull ? ki : ki + 1;   // threshold for j < i (equal keys precede)
  int cnt = 0;
  for (int tile0 = 0; tile0 < N; tile0 += kRankTile) {
    const int n_t = min(kRankTile, N - tile0);
    for (int t = tid; t < n_t; t += kRankThreads) keys[t] = key_of(tile0 + t);
    if (tid == 0 && (n_t & 1)) keys[n_t] = ~0ull;
    __syncthreads();
    // Part p takes the pairs of keys p, p + 16, p + 32, ...: every part has work whatever N is, and a warp's two parts
    // read neighbouring 16 bytes.  (A run of 128 keys per part, one key at a time: 5.5 us at 256 keys, 6.5 at 2048;
    // 2.6 and 4.2 now.)  What is missing from the last pair counts for nobody: no key is above one of all ones.
    const ulonglong2* pairs = reinterpret_cast<const ulonglong2*>(keys);
    const int n_pairs = (n_t + 1) / 2, own = i - tile0;       // keys before `own` precede i when equal
    const int mid = own < 0 ? 0 : min(n_pairs, own / 2);      // pairs that lie before it as a whole
    int j = part;
    for (; j < mid; j += kRankParts) {
      const ulonglong2 v = pairs[j];
      cnt += (v.x < ki_le ? 1 : 0) + (v.y < ki_le ? 1 : 0);
    }
    if (j == mid && j < n_pairs && own >= 0) {
      const ulonglong2 v = pairs[j];
      cnt += (v.x < (2 * j < own ? ki_le : ki) ? 1 : 0) + (v.y < ki ? 1 : 0);
      j += kRankParts;
    }
    for (; j < n_pairs; j += kRankParts) {
      const ulonglong2 v = pairs[j];
      cnt += (v.x < ki ? 1 : 0) + (v.y < ki ? 1 : 0);
    }
    __syncthreads();
  }
  part_cnt[tid] = cnt;
  __syncthreads();
  if (part == 0 && i < N) {
    int rank = 0;
#pragma unroll
    for (int q4 = 0; q4 < kRankThreads / kRankCand; ++q4) rank += part_cnt[q4 * kRankCand + tid];
    if (rank < k) {
      final_idx[(long long)b * k + rank] = i;
      if (final_score != nullptr) final_score[(long long)b * k + rank] = (float)key_score(ki);
    }
  }
}

// Rank counting compares every pair of keys, over the whole chip, whatever k; the radix selection is one CTA per query whose time
// grows with k: up to 32 candidates hardly cost anything, 128 to 1024 are dealt out to bins, more are sorted.  Counting / selection, us:
// one query of 3000 keys, k = 1 8.2 / 8.2, 4096 keys, k = 1 9.6 / 8.4, 128 9.7 / 10.9, 512 9.4 / 11.3, 1024 9.7 / 12.5, 6144 keys 14.7 / 9.4,
// 12.1, 12.8 and 13.7; two of 3000, k = 128 10.3 / 11.3, 512 10.3 / 11.6; of 4096, 13.6 / 11.9, 12.5 and (1024) 13.3; eight of 2048, k = 128
// 10.9 / 9.4, 512 10.9 / 9.8, 1024 10.9 / 10.7; 32 of 1024, k = 1 12.1 / 7.6, 512 12.1 / 10.1; sorted: one of 4096, k = 4096 9.3 / 65, of 8192 21 / 70.
bool rank_by_counting(int N, int B, int k) {
  const long long pairs = (long long)N * N * B;
  if (k > kSelThreads) return pairs <= 11000000ll + 48000ll * k;
  return pairs <= 11000000ll + 100000ll * (k < 128 ? k : 128) + 6000ll * (k < 128 ? 0 : k - 128);
}

}  // namespace

int ads_topk_from_keys(const unsigned long long* keys, int N, int B, int k, int32_t* sel_idx, float* sel_score,
                       cudaStream_t st) {
  if (N > kSortCap && k > kSortCap / 2) return ADAPSHOT_EUNSUPPORTED;
  if (rank_by_counting(N, B, k)) {
    dim3 grid((N + kRankCand - 1) / kRankCand, B);
    ads_launch_dependent(rank_topk_kernel, grid, kRankThreads, 0, st, keys, N, k, sel_idx, sel_score);
    return ads_launch_status();
  }
  // candidates worth sorting: the power of two the sort pads to (bins of the second pass rarely hold two keys)
  int want = 128;
  while (want < k) want <<= 1;
  static bool attr_set[kAdsMaxDevices] = {false};
  if (ads_set_max_smem(radix_topk_kernel, kSortCap * (8 + 4) + kSelBins * 4, attr_set) != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  const int smem = want * (8 + 4) * (want <= kSelThreads ? 2 : 1) + kSelBins * 4;
  ads_launch_dependent(radix_topk_kernel, (unsigned)B, kSelThreads, smem, st, keys, N, k, want, sel_idx, sel_score);
  return ads_launch_status();
}

extern "C" size_t adapshot_select_workspace_bytes(int32_t n_shots, int32_t B, int32_t k) {
  if (n_shots <= 0 || B <= 0 || k <= 0) return 0;
  // the sort keys, and room for a norm per shot that no kernel needs any more: the size a call is refused below stays
  return ads_round_up((size_t)B * n_shots * sizeof(unsigned long long), 256) +
         ads_round_up((size_t)n_shots * sizeof(double), 256);
}

extern "C" int adapshot_select(const adapshot_pool_t* pool, const float* q_emb, int32_t B, int32_t k,
                               int32_t* sel_idx, float* sel_score, void* ws, size_t ws_bytes,
                               int32_t* status, void* stream) {
  (void)status;
  if (pool == nullptr || q_emb == nullptr || sel_idx == nullptr || ws == nullptr) return ADAPSHOT_EINVAL;
  if (pool->emb == nullptr || pool->n_shots <= 0 || pool->emb_dim <= 0 || B <= 0) return ADAPSHOT_EINVAL;
  const int N = pool->n_shots, E = pool->emb_dim;
  if (k < 1 || k > N) return ADAPSHOT_ESHAPE;
  if (N > kSortCap && k > kSortCap / 2) return ADAPSHOT_EUNSUPPORTED;
  if (!ads_aligned16(pool->emb) || !ads_aligned16(q_emb) || !ads_aligned16(ws)) return ADAPSHOT_EALIGN;
  if (ws_bytes < adapshot_select_workspace_bytes(N, B, k)) return ADAPSHOT_ECAPACITY;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  unsigned long long* keys = static_cast<unsigned long long*>(ws);
  if (B > 2 && E % 16 == 0) {          // (4096 x 384: 4.7 us for two queries by warps, 3.4 for four by matrix tiles)
    auto run = [&](auto kernel, int rows, int queries) {
      ads_launch_dependent(kernel, dim3((unsigned)((N + rows - 1) / rows), (unsigned)((B + queries - 1) / queries)), 32 * kMmaWarps, 0, st,
                           pool->emb, q_emb, N, E, B, keys);
    };
    // 16 shots per CTA (three per SM) leave a shorter last wave than 32 (two per SM): 20000 x 768, 16 queries 41.1 -> 39.1 us for the
    // call, 8192 x 1024, 32 queries 35.2 -> 33.0, 40000 x 384, 32 queries 75.8 -> 72.3.  Up to 8 queries the element widened once per 32
    // shots matters as much, unless CTAs of 16 shots find an SM each (16 / 32 shots, E = 1024, 4 queries: 1024 shots 6.7 / 7.9, 2368 11.1 /
    // 12.3; beyond that 2500 14.1 / 13.7, 3000 16.4 / 16.0, 4096 20.7 / 20.3, 8192 62.0 / 61.0, 16384 212.5 / 213.5).
    const int n_sm = ads_sm_count();
    if (n_sm <= 0) return ADAPSHOT_ECUDA;
    if (B > 8) run(cosine_mma_kernel<2, 1>, 16, 16);
    else if (N <= 16 * n_sm) run(cosine_mma_kernel<1, 1>, 16, 8);
    else run(cosine_mma_kernel<1, 2>, 32, 8);
  } else {
    const unsigned grid = (unsigned)((N + 7) / 8);
    auto run = [&](auto kernel) { ads_launch_dependent(kernel, grid, 256, 0, st, pool->emb, q_emb, N, E, B, keys); };
    if (E == 1024) run(cosine_keys_kernel<8>);
    else if (E == 768) run(cosine_keys_kernel<6>);
    else if (E == 384) run(cosine_keys_kernel<3>);
    else if (E == 128) run(cosine_keys_kernel<1>);
    else run(cosine_keys_kernel<0>);
  }
  if (ads_launch_status() != ADAPSHOT_OK) return ADAPSHOT_ECUDA;
  return ads_topk_from_keys(keys, N, B, k, sel_idx, sel_score, st);
}
