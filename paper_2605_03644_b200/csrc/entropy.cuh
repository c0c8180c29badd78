// Device code of the probe entropy, a block at a time: entropy.cu runs it as kernels of its own, a pass in one call
// (attn.cu) beside the attention's small kernels.
#pragma once

#include <float.h>

#include "common.cuh"

namespace {

struct EntState {
  float m, s, t;
};

__device__ __forceinline__ EntState ent_merge(EntState a, EntState b) {
  float M = fmaxf(a.m, b.m);
  float ea = __expf(a.m - M), eb = __expf(b.m - M);
  // a state with s == 0 has seen nothing (or only -inf): it adds nothing
  float ta = a.s > 0.f ? (a.t + a.s * (a.m - M)) * ea : 0.f;
  float tb = b.s > 0.f ? (b.t + b.s * (b.m - M)) * eb : 0.f;
  EntState r;
  r.m = M;
  r.s = a.s * ea + b.s * eb;
  r.t = ta + tb;
  return r;
}

__device__ __forceinline__ float ent_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ent_max3(float a, float b, float c) {   // one instruction on sm_100
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Logits at or below this value count as -inf: the loaders raise every logit to it (an exact
// operation), so that x - m stays finite and e * (x - m) is -0, not NaN, where e underflows to 0.
// -2^97 is exact in bf16 and in fp32.  A row that holds nothing above it has entropy 0 by
// convention (ent_finish_block).
constexpr float kEntFloor = -1.5845632502852868e29f;
constexpr uint32_t kEntFloorBf16x2 = 0xF000F000u;

// A thread's running state: two interleaved sums each, so that pairs of logits go through the two-wide fp32
// instructions and nothing is added across a pair before the end.
struct EntRun {
  float m;
  float2 s, t;
};

// Adds N logits (already raised to kEntFloor) to a state.  d = x - m is formed exactly (the row
// maximum itself gives d = 0 and e = 1), e = 2^(d log2 e) is one multiply and one MUFU operation,
// t accumulates e * d.
template <int N>
__device__ __forceinline__ void ent_accumulate(EntRun& st, const float (&x)[N]) {
  constexpr float kLog2e = 1.4426950408889634f;
  float vm = x[0];
  {
    int i = 1;
#pragma unroll
    for (; i + 1 < N; i += 2) vm = ent_max3(vm, x[i], x[i + 1]);
    if (i < N) vm = fmaxf(vm, x[i]);
  }
  if (vm > st.m) {
    const float d = st.m - vm, e = __expf(d);
    st.t.x = st.s.x > 0.f ? (st.t.x + st.s.x * d) * e : 0.f;
    st.t.y = st.s.y > 0.f ? (st.t.y + st.s.y * d) * e : 0.f;
    st.s.x *= e;
    st.s.y *= e;
    st.m = vm;
  }
  if constexpr (N % 2 == 0) {
    const float2 neg_m = make_float2(-st.m, -st.m), l2e = make_float2(kLog2e, kLog2e);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const float2 d = __fadd2_rn(make_float2(x[i], x[i + 1]), neg_m);
      const float2 a = __fmul2_rn(d, l2e);
      const float2 e = make_float2(ent_ex2(a.x), ent_ex2(a.y));
      st.s = __fadd2_rn(st.s, e);
      st.t = __ffma2_rn(e, d, st.t);
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float d = x[i] - st.m;
      const float e = ent_ex2(d * kLog2e);
      st.s.x += e;
      st.t.x = fmaf(e, d, st.t.x);
    }
  }
}

__device__ __forceinline__ EntState ent_warp_reduce(EntState st) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    EntState other;
    other.m = __shfl_xor_sync(0xffffffffu, st.m, o);
    other.s = __shfl_xor_sync(0xffffffffu, st.s, o);
    other.t = __shfl_xor_sync(0xffffffffu, st.t, o);
    st = ent_merge(st, other);
  }
  return st;
}

constexpr int kEntThreads = 256;

// partial[block] = state of slice s of row r, block = r * n_split + s: a block of kEntThreads.
template <typename T>
__device__ __forceinline__ void ent_partial_block(const T* __restrict__ logits, int V, long long row_stride, int slice,
                                                  int n_split, float* __restrict__ partial, int block) {
  constexpr int kVec = 16 / sizeof(T);
  constexpr float kLog2e = 1.4426950408889634f;
  const int r = block / n_split, sp = block % n_split;
  const T* row = logits + (long long)r * row_stride;
  const int begin = sp * slice;
  const int end = V - begin <= slice ? V : begin + slice;      // (begin + slice may not fit an int)
  EntRun st{kEntFloor, {0.f, 0.f}, {0.f, 0.f}};    // every logit is at least the floor, so m starts there

  const int n_vec = (end - begin) / kVec;                        // slice is a multiple of kVec
  auto widen = [](const uint4& raw, float (&x)[kVec]) {
    if constexpr (sizeof(T) == 4) {
      x[0] = fmaxf(__uint_as_float(raw.x), kEntFloor); x[1] = fmaxf(__uint_as_float(raw.y), kEntFloor);
      x[2] = fmaxf(__uint_as_float(raw.z), kEntFloor); x[3] = fmaxf(__uint_as_float(raw.w), kEntFloor);
    } else {
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {   // the floor on both halves at once; bf16 -> fp32 is a 16-bit shift
        uint32_t c;
        asm("max.bf16x2 %0, %1, %2;" : "=r"(c) : "r"(w[j]), "r"(kEntFloorBf16x2));
        x[2 * j] = __uint_as_float(c << 16);
        x[2 * j + 1] = __uint_as_float(c & 0xffff0000u);
      }
    }
  };
  // Four 16-byte loads per thread are kept in flight: a vector is copied out of its register,
  // the load of the vector four steps ahead goes into that register at once, and only then is
  // the copy worked on, so the memory system is never idle while a warp computes.  The host cuts
  // rows into slices that are multiples of kEntSliceUnit, so that all but a row's last slice run
  // in this loop alone.
  constexpr int kUnroll = 4;
  const uint4* vp = reinterpret_cast<const uint4*>(row + begin) + threadIdx.x;
  const uint4* const vp_end = reinterpret_cast<const uint4*>(row + begin) + n_vec;
  const int trips = n_vec / (kUnroll * kEntThreads);
  if (trips > 0) {
    uint4 raw[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) raw[u] = __ldcs(vp + u * kEntThreads);
    for (int t = 1; t < trips; ++t) {
      vp += kUnroll * kEntThreads;
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        float x[kVec];
        widen(raw[u], x);
        raw[u] = __ldcs(vp + u * kEntThreads);
        ent_accumulate(st, x);
      }
    }
    vp += kUnroll * kEntThreads;
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      float x[kVec];
      widen(raw[u], x);
      ent_accumulate(st, x);
    }
  }
  for (; vp < vp_end; vp += kEntThreads) {
    float x[kVec];
    widen(__ldcs(vp), x);
    ent_accumulate(st, x);
  }
  for (int i = begin + n_vec * kVec + threadIdx.x; i < end; i += kEntThreads) {   // ragged tail of the row
    float x[1];
    if constexpr (sizeof(T) == 4) x[0] = fmaxf(row[i], kEntFloor);
    else x[0] = fmaxf(__bfloat162float(row[i]), kEntFloor);
    ent_accumulate(st, x);
  }

  // CTA-wide merge: the maximum first; every thread then moves its (s, t) to it once, and what is
  // left are plain sums (a butterfly of whole states would pay two exponentials per level)
  __shared__ float sh_m[kEntThreads / 32], sh_s[kEntThreads / 32], sh_t[kEntThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float M = st.m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  if (lane == 0) sh_m[warp] = M;
  __syncthreads();
  M = sh_m[0];
#pragma unroll
  for (int w = 1; w < kEntThreads / 32; ++w) M = fmaxf(M, sh_m[w]);
  const float d = fmaxf(st.m - M, -1.0e30f);          // <= 0; the clamp keeps s * d finite
  const float e = ent_ex2(d * kLog2e);
  const float s_all = st.s.x + st.s.y;
  float ss = s_all * e, tt = fmaf(s_all, d, st.t.x + st.t.y) * e;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    tt += __shfl_xor_sync(0xffffffffu, tt, o);
  }
  if (lane == 0) { sh_s[warp] = ss; sh_t[warp] = tt; }
  __syncthreads();
  if (threadIdx.x == 0) {
    ss = 0.f; tt = 0.f;
#pragma unroll
    for (int w = 0; w < kEntThreads / 32; ++w) { ss += sh_s[w]; tt += sh_t[w]; }
    float* o = partial + 3ll * ((long long)r * n_split + sp);
    o[0] = M; o[1] = ss; o[2] = tt;
  }
}

// A block finishes group g of `rows_per_group` rows: warp w merges the splits of rows w, w + n_warps, ...; thread 0
// then applies the threshold rule to the group.  sh_h: rows_per_group floats of shared memory.
__device__ __forceinline__ void ent_finish_block(const float* __restrict__ partial, int n_split, int R, int rows_per_group,
                                                 float tau, float* __restrict__ H, int32_t* __restrict__ first_ok, int g,
                                                 float* sh_h) {
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
    if (lane == 0) {
      // a maximum at the floor: the row holds nothing but -inf (or values that count as it)
      float h = (st.s > 0.f && st.m > kEntFloor) ? logf(st.s) - st.t / st.s : 0.f;
      h = fmaxf(h, 0.f);
      H[r] = h;
      sh_h[j] = h;
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

}  // namespace
