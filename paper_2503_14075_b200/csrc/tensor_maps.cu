// Tensor maps (TMA) over the K / V cache and a call's tree rows, for the tcgen05 tree-attention kernels.
#include <cuda.h>

#include <mutex>

#include "tree_attn.cuh"

namespace twig {

// ---- tensor maps over the whole K and V cache: dims (d, pos, head, batch, layer) ----
namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct MapKey {
  const void *k, *v;
  long long sl, sb, sh, sp;
  int n_layers, batch, heads, max_len, head_dim, box_rows;
  bool operator==(const MapKey &o) const {
    return k == o.k && v == o.v && sl == o.sl && sb == o.sb && sh == o.sh && sp == o.sp && n_layers == o.n_layers &&
           batch == o.batch && heads == o.heads && max_len == o.max_len && head_dim == o.head_dim && box_rows == o.box_rows;
  }
};
struct MapEntry {
  MapKey key;
  alignas(64) CUtensorMap kmap;
  alignas(64) CUtensorMap vmap;
  bool valid = false;
};
constexpr int kMapEntries = 32;      // (a cache in use takes up to three entries)

static EncodeTiledFn encode_tiled() {
  static const EncodeTiledFn fn = []() -> EncodeTiledFn {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    const bool found = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
                       qres == cudaDriverEntryPointSuccess;
    return found ? reinterpret_cast<EncodeTiledFn>(ptr) : nullptr;
  }();
  return fn;
}

static bool encode_cache_map(EncodeTiledFn fn, CUtensorMap *out, const void *base, const MapKey &key) {
  const cuuint64_t dims[5] = {(cuuint64_t)key.head_dim, (cuuint64_t)key.max_len, (cuuint64_t)key.heads, (cuuint64_t)key.batch,
                              (cuuint64_t)key.n_layers};
  const cuuint64_t strides[4] = {(cuuint64_t)key.sp * 2, (cuuint64_t)key.sh * 2, (cuuint64_t)key.sb * 2,
                                 (cuuint64_t)key.sl * 2};
  const cuuint32_t box[5] = {64, (cuuint32_t)key.box_rows, 1, 1, 1};   // 128 bytes x KT rows: one swizzled panel
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Copies the (cached) pair of maps for this cache layout into `out`; false when none can be made.
// (The table is a small ring that other threads may overwrite as soon as the lock is gone, so
// the caller gets a copy, not a pointer into it.)
bool cache_maps(const AttnParams &p, int box_rows, CacheMaps *out) {
  static std::mutex mu;
  static MapEntry table[kMapEntries];
  static int next = 0;
  const EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  std::lock_guard<std::mutex> lock(mu);
  // strides must be multiples of 16 bytes, and every dimension but the last needs stride * extent in range
  if (p.c_sp <= 0 || p.c_sh <= 0 || p.c_sb < 0 || p.c_sl < 0) return false;
  MapKey key{p.cache_k0, p.cache_v0, p.n_layers > 1 ? p.c_sl : p.c_sp, p.batch > 1 ? p.c_sb : p.c_sp, p.c_sh, p.c_sp,
             p.n_layers, p.batch, p.n_kv_heads, p.max_len, p.head_dim, box_rows};
  if (p.n_kv_heads == 1) key.sh = key.sp;      // a stride of an extent-1 dimension is never used
  for (auto &e : table)
    if (e.valid && e.key == key) {
      out->kmap = e.kmap;
      out->vmap = e.vmap;
      return true;
    }
  MapEntry &e = table[next];
  next = (next + 1) % kMapEntries;
  e.valid = false;
  if (!encode_cache_map(fn, &e.kmap, p.cache_k0, key) || !encode_cache_map(fn, &e.vmap, p.cache_v0, key)) return false;
  e.key = key;
  e.valid = true;
  out->kmap = e.kmap;
  out->vmap = e.vmap;
  return true;
}

bool tree_maps(const AttnParams &p, int box_rows, CacheMaps *out) {
  const EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)p.head_dim, (cuuint64_t)p.t_max, (cuuint64_t)p.batch * p.n_kv_heads};
  const cuuint64_t strides[2] = {(cuuint64_t)p.head_dim * 2, (cuuint64_t)p.head_dim * 2 * p.t_max};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1}, estr[3] = {1, 1, 1};
  auto encode = [&](CUtensorMap *map, const __nv_bfloat16 *base) {
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16 *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  return encode(&out->kmap, p.tree_k) && encode(&out->vmap, p.tree_v);
}

}  // namespace twig
