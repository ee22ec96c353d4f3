// One pass over a row of logits (a distribution over the vocabulary), split between the CTAs of a cluster.
//
// A row is 64 to 500 KB and a call has few rows (one per request or tree node), so what bounds the pass is the
// chain of load latencies of one CTA, not the bandwidth: a row is cut into slices for up to eight CTAs, each
// thread has all of its 16-byte loads of a batch in flight, and per 16-byte chunk only the maximum is
// compared; the winning chunk is kept in registers and the element looked up in it at the end.
#pragma once

#include <cooperative_groups.h>

#include "tree_attn.cuh"

namespace twig {

constexpr int kRowThreads = 256;
constexpr int kRowDeep = 8;            // 16-byte loads in flight per thread
constexpr int kMaxSlices = 8;

// (maximum, its index (the lowest of equals), sum of exp(x - maximum))
struct RowBest {
  float m, s;
  int index;
};

template <bool FP32>
struct RowFormat {
  static constexpr int EPC = FP32 ? 4 : 8;         // elements per chunk
  static __device__ __forceinline__ void unpack(const uint4 &w, float (&v)[EPC]) {
    if constexpr (FP32) {
      v[0] = __uint_as_float(w.x); v[1] = __uint_as_float(w.y); v[2] = __uint_as_float(w.z); v[3] = __uint_as_float(w.w);
    } else {
      v[0] = bf16_lo(w.x); v[1] = bf16_hi(w.x); v[2] = bf16_lo(w.y); v[3] = bf16_hi(w.y);
      v[4] = bf16_lo(w.z); v[5] = bf16_hi(w.z); v[6] = bf16_lo(w.w); v[7] = bf16_hi(w.w);
    }
  }
  static __device__ __forceinline__ float element(const unsigned char *row, int i) {
    return FP32 ? reinterpret_cast<const float *>(row)[i] : __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(row)[i]);
  }
  // the chunk that holds the row's tail (vocab no multiple of EPC), read by elements, -inf past the end
  static __device__ __forceinline__ void tail(const unsigned char *row, int chunk, int vocab, float (&v)[EPC]) {
#pragma unroll
    for (int e = 0; e < EPC; ++e) v[e] = chunk * EPC + e < vocab ? element(row, chunk * EPC + e) : -INFINITY;
  }
};

template <bool SUM>
__device__ __forceinline__ void row_merge(RowBest &a, float m, float s, int index) {
  const float top = fmaxf(a.m, m);
  if (SUM) {
    const float ref = top == -INFINITY ? 0.f : top;
    a.s = a.s * __expf(a.m - ref) + s * __expf(m - ref);
  }
  if (m > a.m || (m == a.m && index < a.index)) a.index = index;
  a.m = top;
}

// This CTA's slice of the row: chunks first, first + 1, .. below last (whole chunks), and the tail chunk when
// `with_tail`.  Every thread returns the CTA's result in warp 0.
template <bool FP32, bool SUM>
__device__ __forceinline__ RowBest scan_slice(const unsigned char *row, int first, int last, bool with_tail, int vocab) {
  using F = RowFormat<FP32>;
  __shared__ RowBest s_part[kRowThreads / 32];
  const int tid = threadIdx.x;
  RowBest best{-INFINITY, 0.f, 0x7fffffff};
  uint4 top = make_uint4(0u, 0u, 0u, 0u);          // the chunk that holds the maximum, and its number
  int at = -1;
  for (int c0 = first + tid; c0 < last; c0 += kRowDeep * kRowThreads) {
    uint4 w[kRowDeep];
#pragma unroll
    for (int u = 0; u < kRowDeep; ++u)
      if (c0 + u * kRowThreads < last) w[u] = ld_nc_16(row + (long long)(c0 + u * kRowThreads) * 16);
    float m = best.m;
    if (at < 0) {                                  // (so that a row of -inf has an index)
      at = c0;
      top = w[0];
    }
#pragma unroll
    for (int u = 0; u < kRowDeep; ++u)
      if (c0 + u * kRowThreads < last) {
        float v[F::EPC];
        F::unpack(w[u], v);
        float cm = v[0];
#pragma unroll
        for (int e = 1; e < F::EPC; ++e) cm = fmaxf(cm, v[e]);
        if (cm > m) {
          at = c0 + u * kRowThreads;
          top = w[u];
        }
        m = fmaxf(m, cm);
      }
    if (SUM) {
      const float ref = m == -INFINITY ? 0.f : m;
      float s = best.s * __expf(best.m - ref), t = 0.f;
#pragma unroll
      for (int u = 0; u < kRowDeep; ++u)
        if (c0 + u * kRowThreads < last) {
          float v[F::EPC];
          F::unpack(w[u], v);
#pragma unroll
          for (int e = 0; e < F::EPC; e += 2) {
            s += __expf(v[e] - ref);
            t += __expf(v[e + 1] - ref);
          }
        }
      best.s = s + t;
    }
    best.m = m;
  }
  if (at >= 0) {
    float v[F::EPC];
    F::unpack(top, v);
#pragma unroll
    for (int e = F::EPC - 1; e >= 0; --e)
      if (v[e] == best.m) best.index = at * F::EPC + e;
  }
  if (with_tail && tid == 0) {
    float v[F::EPC], m = -INFINITY, s = 0.f;
    F::tail(row, vocab / F::EPC, vocab, v);
#pragma unroll
    for (int e = 0; e < F::EPC; ++e) m = fmaxf(m, v[e]);
    if (SUM && m > -INFINITY)
#pragma unroll
      for (int e = 0; e < F::EPC; ++e) s += __expf(v[e] - m);
    int index = vocab / F::EPC * F::EPC;
#pragma unroll
    for (int e = F::EPC - 1; e >= 0; --e)
      if (v[e] == m && vocab / F::EPC * F::EPC + e < vocab) index = vocab / F::EPC * F::EPC + e;
    row_merge<SUM>(best, m, s, index);
  }
  auto over_lanes = [&](int from) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (o > from) continue;
      const float m = __shfl_xor_sync(0xffffffffu, best.m, o), s = SUM ? __shfl_xor_sync(0xffffffffu, best.s, o) : 0.f;
      const int c = __shfl_xor_sync(0xffffffffu, best.index, o);
      row_merge<SUM>(best, m, s, c);
    }
  };
  over_lanes(16);
  if ((tid & 31) == 0) s_part[tid >> 5] = best;
  __syncthreads();
  if (tid < 32) {
    best = (tid & 31) < kRowThreads / 32 ? s_part[tid & 31] : RowBest{-INFINITY, 0.f, 0x7fffffff};
    over_lanes(kRowThreads / 64);
    best.m = __shfl_sync(0xffffffffu, best.m, 0);
    best.s = __shfl_sync(0xffffffffu, best.s, 0);
    best.index = __shfl_sync(0xffffffffu, best.index, 0);
  }
  return best;
}

// The slices of a cluster.  start() comes after every exit that is uniform over the cluster and before the scan;
// merge() returns the row's result in warp 0 of the cluster's first CTA (false there: a peer never delivered).
struct SliceMerge {
  float4 *peer;                // [kMaxSlices], shared
  uint32_t bar;
  int rank, slices;

  __device__ __forceinline__ void start() {
    if (slices == 1) return;
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      mbar_arrive_expect_tx(bar, (uint32_t)(slices - 1) * 16);
      mbar_init_fence_cluster();
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }
  template <bool SUM>
  __device__ __forceinline__ bool merge(RowBest &best) {
    if (slices == 1) return true;
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // every CTA is running, its barrier is set up
    if (rank > 0) {
      if (threadIdx.x == 0)
        st_async_f32x4(map_to_cta(smem_u32(peer + rank), 0), best.m, best.s, __int_as_float(best.index), 0.f, map_to_cta(bar, 0));
      return true;
    }
    if (threadIdx.x >= 32) return true;
    bool landed = mbar_try_wait(bar, 0);
    if (!landed) {
      unsigned long long t0, t1;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
      do {                                         // at most 0.2 s
        landed = mbar_try_wait(bar, 0);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
      } while (!landed && t1 - t0 < 200000000ull);
    }
    for (int r = 1; r < slices; ++r) {
      const float4 o = peer[r];
      row_merge<SUM>(best, o.x, o.y, __float_as_int(o.z));
    }
    return landed;
  }
};

// CTAs per row: enough slices to put all of the rows' loads in flight at once, while the slices of all rows
// fit two CTAs per SM and a slice keeps a chunk per thread
inline int row_slices(long long rows, int chunks) {
  int s = 1;
  while (s < kMaxSlices && rows * s * 2 <= 2 * 148 && chunks >= 2 * s * kRowThreads) s *= 2;
  return s;
}

}  // namespace twig
