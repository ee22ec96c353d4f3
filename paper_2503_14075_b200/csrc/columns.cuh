// Helpers for accumulators read by column: a lane of tensor memory is a key (a row of the instruction's M side),
// a column a query row, so what belongs to a query row is spread over the lanes of four warps.
#pragma once

#include "tcgen05_common.cuh"

namespace twig {

template <int N>
__device__ __forceinline__ void tmem_load(uint32_t taddr, uint32_t (&v)[N]) {
  static_assert(N == 8 || N == 16 || N == 32, "");
  if constexpr (N == 32) {
    tmem_ld32(taddr, v);
  } else if constexpr (N == 16) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(taddr));
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
  }
  tmem_ld_wait();
}
template <int N>
__device__ __forceinline__ void tmem_store(uint32_t taddr, const uint32_t (&v)[N]) {
  if constexpr (N == 32) {
    tmem_st32(taddr, v);
  } else if constexpr (N == 16) {
    tmem_st16(taddr, v);
  } else {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
  }
  tmem_st_wait();
}

// N values per lane -> one per lane: lane i ends with op over the warp of value i / (32 / N)
template <int N, class Op>
__device__ __forceinline__ float column_reduce(float (&v)[N], int lane, Op op) {
  int o = 16;
#pragma unroll
  for (int w = N / 2; w >= 1; w >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float keep = up ? v[i + w] : v[i], send = up ? v[i] : v[i + w];
      v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  }
#pragma unroll
  for (; o >= 1; o >>= 1) v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
  return v[0];
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// barrier that also tells every thread whether any of them said so
__device__ __forceinline__ bool bar_any(int id, int threads, bool mine) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(any)
      : "r"((uint32_t)mine), "r"(id), "r"(threads)
      : "memory");
  return any != 0;
}
// maximum over the warp
__device__ __forceinline__ float warp_max(float x) {
  float y;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace twig
