// K / V tiles of 128 keys for the tcgen05 tree-attention kernels: the tensor maps and the loads of one
// warp.  Key positions: cached prefix row j at j, tree node j at L8 + j with L8 the prefix length
// rounded up to 8, so that every row comes in whole TMA boxes; the gap is masked.
#pragma once

#include "tcgen05_common.cuh"

namespace twig {

constexpr int kTileKeys = 128;
constexpr int kPanelBytes = kTileKeys * 128;       // 64 columns of a K (or V) tile, 128-byte swizzle
template <int D>
__host__ __device__ constexpr int tile_bytes() { return D / 64 * kPanelBytes; }

// K and V: the cache in boxes of 128, 32 and 8 rows, the tree's rows in boxes of 8
struct TileMaps {
  CacheMaps whole, box32, box8, tree8;
};
inline bool tile_maps(const AttnParams &p, TileMaps *m) {
  return cache_maps(p, kTileKeys, &m->whole) && cache_maps(p, 32, &m->box32) && cache_maps(p, 8, &m->box8) &&
         tree_maps(p, 8, &m->tree8);
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// one box of a 3-D tensor map (x, node, request x head)
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int node, int slice) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(node), "r"(slice) : "memory");
}

// Where a tile comes from: one (request, kv head) of the call.
struct TileSource {
  int L, L8, NK;                // cached prefix rows, rounded up to 8, end of the tree's rows
  int hk, b, layer, slice;      // slice: b * n_kv_heads + hk
};

// A tile that lies in the cached prefix: a box per panel.  Every lane arrives once on `bar` (count 32).
template <int D>
__device__ __forceinline__ void load_whole_tile(const TileMaps &maps, const TileSource &s, bool value, uint32_t dst,
                                                uint32_t bar, int k0, int lane) {
  if (lane == 0) {
    const CUtensorMap *map = value ? &maps.whole.vmap : &maps.whole.kmap;
    mbar_arrive_expect_tx(bar, tile_bytes<D>());
    tma_load_5d(dst, map, bar, 0, k0, s.hk, s.b, s.layer);
    if (D == 128) tma_load_5d(dst + kPanelBytes, map, bar, 64, k0, s.hk, s.b, s.layer);
  } else {
    mbar_arrive(bar);
  }
}

// The tile that holds the prefix end and / or tree rows: boxes of 32 and 8 rows spread over the lanes (16-byte
// cp.async cost one warp 1.3 us to issue).  Rows of V between the prefix end and the tree, and after the
// tree up to the next multiple of 16 (the product's step in keys), must be zero: they are cleared once the
// boxes have landed on `bar_raw` (count 1).  Every lane arrives once on `bar`; false: the wait ran out.
template <int D>
__device__ __forceinline__ bool load_edge_tile(const TileMaps &maps, const TileSource &s, bool value, uint32_t dst,
                                               uint32_t bar, uint32_t bar_raw, uint32_t &raw_phase, int k0, int lane,
                                               volatile int *fail) {
  const int pre = min(max(s.L8 - k0, 0), kTileKeys), tree0 = max(k0 - s.L8, 0);
  const int n_tree = min(kTileKeys - pre, s.NK - s.L8 - tree0);
  const uint32_t on = value ? bar_raw : bar;
  const int e1 = pre >> 5, e2 = e1 + ((pre & 31) >> 3), e3 = e2 + ((n_tree + 7) >> 3);
  if (lane == 0) {
    const uint32_t bytes = (uint32_t)(pre + ((n_tree + 7) & ~7)) * (D * 2);
    if (value) mbar_arrive_expect_tx(on, bytes);
    else mbar_expect_tx(on, bytes);
  }
  __syncwarp();
  constexpr int PANELS = D / 64, CPR = D / 8;      // 16-byte chunks per row
  for (int i = lane; i < PANELS * e3; i += 32) {   // every panel of each box
    const int x = i % PANELS * 64, j = i / PANELS;
    const uint32_t to = dst + i % PANELS * kPanelBytes;
    if (j < e2) {
      const int r = j < e1 ? 32 * j : (pre & ~31) + 8 * (j - e1);
      const CacheMaps &m = j < e1 ? maps.box32 : maps.box8;
      tma_load_5d(to + r * 128, value ? &m.vmap : &m.kmap, on, x, k0 + r, s.hk, s.b, s.layer);
    } else {
      const int r = 8 * (j - e2);
      tma_load_3d(to + (pre + r) * 128, value ? &maps.tree8.vmap : &maps.tree8.kmap, on, x, tree0 + r, s.slice);
    }
  }
  bool landed = true;
  if (value) {
    landed = mbar_wait(bar_raw, raw_phase, fail);
    raw_phase ^= 1;
    const int g0 = min(max(s.L - k0, 0), kTileKeys), t0 = pre + n_tree, t1 = min(kTileKeys, (t0 + 15) & ~15);
    for (int i = lane; i < (pre - g0 + t1 - t0) * CPR; i += 32) {
      const int q = i / CPR, r = q < pre - g0 ? g0 + q : t0 + q - (pre - g0);
      asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(dst + (i % CPR >> 3) * kPanelBytes + r * 128 + (i & 7) * 16), "r"(0u) : "memory");
    }
    fence_async_smem();
  }
  mbar_arrive(bar);
  return landed;
}

}  // namespace twig
