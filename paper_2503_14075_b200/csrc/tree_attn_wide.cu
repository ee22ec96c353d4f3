// Tree attention for more than 64 query rows per kv head (grouped-query models) on the 5th-generation
// tensor cores.  Here the tensor cores and the exponentials are the bound (448 rows: 448 flops a byte),
// so the kernel keeps two independent streams of (product, softmax, product) in flight in every CTA: while
// the softmax of one stream runs, the tensor cores work on the other.
//
// A stream is a 128-row accumulator in tensor memory (S 128 columns, O 128 columns; two streams fill it) and
// four softmax warps, one row per thread: row maxima and sums need no exchange at all.  P goes back to tensor
// memory over the first half of its S tile as the A operand of O += P V.
//   more than 128 rows in the block: the streams are the two halves of up to 256 rows, every K / V tile serves both;
//   up to 128 rows: both streams hold the same rows, each takes every other key tile, and their
//     partial results are added at the end.
//
// Warps 0-3 and 4-7: softmax of stream 0 and 1 (they also load Q); warp 8: loader, K and V tiles of 128 keys by
// TMA into a ring of five 32 KB slots; warp 9: one thread issues all products.
// Key splits of a cluster are merged through distributed shared memory: every thread sends its row's
// (m, l) and O / l as scaled fp16 to the row's owner.
// Every wait is bounded: if one runs out the request is flagged TWIG_DEV_INTERNAL.
#include <cooperative_groups.h>
#include <cuda.h>

#include "attn_tiles.cuh"

namespace cg = cooperative_groups;

namespace twig {

namespace {

constexpr int kD = 128;                            // head_dim
constexpr int kTileBytes = tile_bytes<kD>();
constexpr int kKeys = kTileKeys;
constexpr int kRows = 256;                         // rows of a CTA: two streams of 128
constexpr int kThreads = 384;                      // three warpgroups: registers are shared out between whole ones
constexpr int kSlots = 5;
constexpr int kPreUnits = 2;                       // units requested before the predecessor is waited for
constexpr int kPolyOf = 4;
constexpr float kLazyMax = 8.f;                    // raise the running max only beyond this (log2 units)
constexpr int kQBytes = 128 * kD * 2;              // Q of one stream: two 64-column panels of 128 x 128 B
constexpr int kRingBytes = kSlots * kTileBytes;
constexpr int kSmemBytes = 2 * kQBytes + kRingBytes;
constexpr uint32_t kTmemCols = 512;                // S of stream i: columns 128 i ..; O: 256 + 128 i ..
static_assert(kRows * kD * 2 <= kRingBytes && kRows * 16 <= 2 * kQBytes, "the split merge receives in the ring and in Q's place");

__global__ void __launch_bounds__(kThreads, 1)
tree_attn_wide_kernel(const AttnParams p, const __grid_constant__ TileMaps maps) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ unsigned long long s_mask[TWIG_MAX_NODES];       // ancestors-or-self of every node
  __shared__ int s_par[TWIG_MAX_NODES];
  __shared__ float2 s_pair[128];                              // (m, l) of stream 1's rows (same rows in both streams)
  // full[kSlots], empty[kSlots], s[2], p[2 streams][2 halves], q[2], o[2], recv, raw
  __shared__ __align__(8) unsigned long long s_bar[2 * kSlots + 12];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;

  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);     // (uniform for the compiler too: see umma8_kk)
  const int split = blockIdx.x, n_splits = gridDim.x;
  const int hk = blockIdx.y / p.row_blocks, rb = blockIdx.y % p.row_blocks;
  const int b = blockIdx.z;

  const uint32_t q_s = smem_u32(smem);
  const uint32_t ring_s = q_s + 2 * kQBytes;
  const uint32_t bars = smem_u32(s_bar);
  auto bar_full = [&](int slot) { return bars + 8 * slot; };
  auto bar_empty = [&](int slot) { return bars + 8 * (kSlots + slot); };
  auto bar_s = [&](int i) { return bars + 8 * (2 * kSlots + i); };
  auto bar_p = [&](int i, int h) { return bars + 8 * (2 * kSlots + 2 + 2 * i + h); };
  auto bar_q = [&](int i) { return bars + 8 * (2 * kSlots + 6 + i); };
  auto bar_o = [&](int i) { return bars + 8 * (2 * kSlots + 8 + i); };
  const uint32_t bar_recv = bars + 8 * (2 * kSlots + 10), bar_raw = bars + 8 * (2 * kSlots + 11);

  // ---- what needs nothing from global memory ----
  if (tid == 0) {
    s_fail = 0;
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(bar_full(i), 32);                  // every loader lane arrives once per unit
      mbar_init(bar_empty(i), 1);                  // one tcgen05.commit
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_s(i), 1);
      mbar_init(bar_p(i, 0), 4);                   // the stream's softmax warps
      mbar_init(bar_p(i, 1), 4);
      mbar_init(bar_q(i), 4);
      mbar_init(bar_o(i), 1);
    }
    mbar_init(bar_recv, 1 + 8);                    // the peers' bytes are announced; this CTA's own share by its softmax warps
    mbar_init(bar_raw, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp == 8 && lane < 8)
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.whole.kmap + lane)) : "memory");
  auto wait_predecessor = [&]() { asm volatile("griddepcontrol.wait;" ::: "memory"); };
  // every exit before the key loop: the dependency is carried on, the tensor memory is handed back
  auto leave = [&]() {
    wait_predecessor();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kTmemCols) : "memory");
  };

  // With `early_prefix` the lengths, the parents and the cached prefix may be read while the preceding
  // kernel drains; q, the tree's rows and the output only after it has completed.
  if (!p.early_prefix) wait_predecessor();
  const int n = p.n_nodes[b], L = p.kv_len[b];
  const int my_parent = tid < p.t_max ? p.parent[(long long)b * p.t_max + tid] : -1;
  const bool first = split == 0 && blockIdx.y == 0 && tid == 0;
  const int rows_total = n * p.group, row0 = rb * kRows;
  if (n <= 0 || n > p.t_max || L < 0 || L > p.max_len || row0 >= rows_total) {
    if (first && (n < 0 || n > p.t_max)) flag_status(p.dev_status, b, TWIG_DEV_BAD_TREE);
    else if (first && n > 0 && (L < 0 || L > p.max_len)) flag_status(p.dev_status, b, TWIG_DEV_OVERFLOW);
    leave();
    return;
  }
  const bool two = rows_total - row0 > 128;        // the streams hold different rows (else: alternate tiles of the same)
  const int L8 = (L + 7) & ~7, NK = L8 + n;
  const int n_tiles = (NK + kKeys - 1) / kKeys;
  const int per = (n_tiles + n_splits - 1) / n_splits;
  const int t_begin = min(n_tiles, split * per);
  const int n_my = min(n_tiles, t_begin + per) - t_begin;

  bool bad = false;
  if (tid < n) {
    s_par[tid] = my_parent;
    bad = (tid == 0) ? (my_parent != -1) : (my_parent < 0 || my_parent >= tid);
  }
  if (__syncthreads_or(bad)) {                     // (also: the barriers are visible)
    if (first) flag_status(p.dev_status, b, TWIG_DEV_BAD_TREE);
    leave();
    return;
  }

  // ---- loader units in the order of their first use: K0 V0 K1 V1 .. with different rows in the streams,
  // K0 K1 V0 K2 V1 .. with alternate tiles ----
  const int n_units = 2 * n_my;
  auto unit_is_v = [&](int u) { return two ? (u & 1) != 0 : u > 0 && (!(u & 1) || u == n_units - 1); };
  auto unit_key = [&](int u) {
    const int t = two ? u >> 1 : u == n_units - 1 ? n_my - 1 : (u & 1) ? (u + 1) >> 1 : u == 0 ? 0 : (u >> 1) - 1;
    return (t_begin + t) * kKeys;
  };
  auto k_unit = [&](int t) { return two ? 2 * t : t == 0 ? 0 : 2 * t - 1; };
  auto v_unit = [&](int t) { return two ? 2 * t + 1 : t == n_my - 1 ? n_units - 1 : 2 * t + 2; };
  const TileSource source{L, L8, NK, hk, b, p.layer, b * p.n_kv_heads + hk};
  auto load_whole = [&](int u) {
    load_whole_tile<kD>(maps, source, unit_is_v(u), ring_s + u % kSlots * kTileBytes, bar_full(u % kSlots), unit_key(u), lane);
  };
  const int n_first = min(n_units, kPreUnits);
  if (warp == 8)
    for (int u = 0; u < n_first; ++u)
      if (unit_key(u) + kKeys <= L) load_whole(u);

  if (tid < n) {                                   // ancestor-or-self bitmask; parent[x] < x bounds the walk
    unsigned long long m = 0;
    for (int x = tid; x >= 0; x = s_par[x]) m |= 1ull << x;
    s_mask[tid] = m;
  }
  // (the loader needs neither the tensor memory nor the masks)
  tc_fence_before();
  if (warp < 8 || warp == 9) asm volatile("bar.sync 1, %0;" ::"n"(9 * 32) : "memory");
  tc_fence_after();
  // (only now, with this CTA's tensor memory allocated, may CTAs of the next kernel be scheduled: they
  // could take the columns and then wait for this kernel to complete)
  wait_predecessor();
  if (warp != 8) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem = s_tmem;
  volatile int *fail = &s_fail;
  const int stream = (warp >> 2) & 1;
  const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);     // this warp's 32 lanes
  const int row_local = two ? tid & 255 : tid & 127;          // softmax threads: their row of the block
  const int gr = row0 + row_local;
  const bool row_valid = warp < 8 && gr < rows_total;
  float m_run = -INFINITY, l_run = 0.f;            // m_run: scaled logits in log2 units

  // (168 registers a thread at launch; a softmax thread holds a row of 128 logits: 2 x 208 + 88 = 3 x 168)
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    if (warp == 8) {
    // ================= loader =================
    uint32_t raw_phase = 0;
    bool ok = true;
    for (int u = 0; u < n_units && ok; ++u) {
      const bool whole = unit_key(u) + kKeys <= L;
      if (u < n_first && whole) continue;          // requested above
      if (u >= kSlots) {
        ok = mbar_wait(bar_empty(u % kSlots), (u / kSlots - 1) & 1, fail);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
      }
      if (whole) {
        load_whole(u);
      } else {
        ok = load_edge_tile<kD>(maps, source, unit_is_v(u), ring_s + u % kSlots * kTileBytes, bar_full(u % kSlots), bar_raw,
                            raw_phase, unit_key(u), lane, fail);
        ok = __all_sync(0xffffffffu, ok);
      }
    }
    if (!ok) s_fail = 1;
    } else if (warp == 9) {
    // ================= MMA issuer (one elected lane; the warp stays together) =================
    if (n_my > 0) {
      const uint32_t leader = elect_one();
      constexpr uint32_t kIdescS = instr_desc(128, kKeys, false), kIdescO = instr_desc(128, kD, true);
      bool ok = true;
      auto wait_full = [&](int u) {
        if (ok) ok = mbar_wait(bar_full(u % kSlots), (u / kSlots) & 1, fail);
      };
      // step k: stream k & 1, its tile
      const int n_steps = two ? 2 * n_my : n_my;
      auto tile_of = [&](int k) { return two ? k >> 1 : k; };
      auto issue_s = [&](int k) {                  // S = Q K^T of step k
        const int i = k & 1, u = k_unit(tile_of(k));
        if (!two || i == 0) wait_full(u);
        if (!ok) return;
        umma8_kk<kPanelBytes, kPanelBytes>(leader, tmem + i * 128, smem_desc(q_s + (two ? i * kQBytes : 0), 16),
                                           smem_desc(ring_s + (u % kSlots) * kTileBytes, 16), kIdescS);
        umma_commit_if(leader, bar_s(i));
        if (!two || i == 1) umma_commit_if(leader, bar_empty(u % kSlots));
      };
      ok = mbar_wait(bar_q(0), 0, fail);
      if (ok && two) ok = mbar_wait(bar_q(1), 0, fail);
      if (ok) issue_s(0);
      if (ok && n_steps > 1) issue_s(1);
      for (int k = 0; k < n_steps && ok; ++k) {
        const int i = k & 1, t = tile_of(k), u = v_unit(t);
        // P arrives in two halves of 64 keys: the product of the first runs while the softmax warps are still at
        // the second (one piece: 3530 cycles per 128 keys of both streams)
        ok = mbar_wait(bar_p(i, 0), (k >> 1) & 1, fail);
        if (!two || i == 0) wait_full(u);
        tc_fence_after();
        if (!ok) break;
        const uint64_t vd = smem_desc(ring_s + (u % kSlots) * kTileBytes, kPanelBytes);
        const int steps = (min(kKeys, NK - (t_begin + t) * kKeys) + 15) >> 4;     // 16 keys each
        const uint32_t o = tmem + 256 + i * 128, pt = tmem + i * 128;
        auto product = [&](int h) {
          if (steps >= 4 * h + 4) umma4_ts<2048>(leader, o, pt + h * 32, vd + h * 512, kIdescO, k > 1 || h > 0);
          else
            for (int j = 4 * h; j < steps; ++j)
              if (leader) umma_ts(o, pt + j * 8, vd + j * 128, kIdescO, k > 1 || j > 0);
        };
        product(0);
        ok = mbar_wait(bar_p(i, 1), (k >> 1) & 1, fail);
        tc_fence_after();
        if (!ok) break;
        product(1);
        if (k + 2 >= n_steps) umma_commit_if(leader, bar_o(i));          // the stream's last product
        if (!two || i == 1) umma_commit_if(leader, bar_empty(u % kSlots));
        if (k + 2 < n_steps) issue_s(k + 2);
      }
      if (!ok && lane == 0) s_fail = 1;
    }
    }
    // the registers come back only once the softmax warps have handed theirs in: a warp that took them before
    // those had grown would make them wait for good
    __syncwarp();
    asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
    asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    // ================= softmax: one row per thread =================
    bool ok = true;
    const bool loads_q = two || stream == 0;
    if (n_my > 0 && loads_q) {                     // Q of this stream (zero rows past the request's last row)
      const int first_row = row0 + (two ? stream * 128 : 0), t128 = tid & 127;
      // (rows stay far below 2^20, so the quotient by multiplication is exact)
      const float inv_group = 1.f / (float)p.group;
#pragma unroll 4
      for (int i = 0; i < 16; ++i) {
        const int r = i * 8 + (t128 >> 4), c = t128 & 15;
        const bool valid = first_row + r < rows_total;
        const int row = valid ? first_row + r : 0, node = (int)(((float)row + 0.5f) * inv_group), g = row - node * p.group;
        const __nv_bfloat16 *src = p.q + (((long long)b * p.t_max + node) * p.n_q_heads + hk * p.group + g) * kD + c * 8;
        cp_async_16(q_s + (two ? stream * kQBytes : 0) + (c >> 3) * kPanelBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4), src, valid);
      }
      cp_async_commit();
      cp_async_wait<0>();
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_q(stream));
    }
    const int n_mine = two ? n_my : (n_my - stream + 1) >> 1;
    const bool warp_idle = row0 + (row_local & ~31) >= rows_total;       // (uniform) no row of this warp exists
    const unsigned long long mask = row_valid ? s_mask[gr / p.group] : 0ull;
    // bit j: key base + j is visible (prefix rows; tree rows by the ancestor mask; not the gap between them)
    auto visible = [&](int base) {
      const int pre = L - base, rel = base - L8;
      unsigned long long v = pre >= 64 ? ~0ull : pre > 0 ? (1ull << pre) - 1ull : 0ull;
      if (rel >= 0) v |= rel < 64 ? mask >> rel : 0ull;
      else if (rel > -64) v |= mask << -rel;
      return v;
    };
    const uint32_t ts = t_lane + stream * 128, to = t_lane + 256 + stream * 128;
    const float sc = p.scale_log2;
    for (int j = 0; j < n_mine; ++j) {
      const int base = (t_begin + (two ? j : 2 * j + stream)) * kKeys;
      ok = ok && mbar_wait(bar_s(stream), j & 1, fail);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      if (!warp_idle) {
        uint32_t s[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(ts + 32 * c, s[c]);
        tmem_ld_wait();
        if (base + kKeys > L) {                    // the prefix end and / or the tree: mask
          const unsigned long long v0 = visible(base), v1 = visible(base + 64);
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (!(((c < 2 ? v0 : v1) >> (32 * (c & 1) + i)) & 1ull)) s[c][i] = 0xff800000u;     // -inf
        }
        float mx[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          mx[c] = fmaxf(__uint_as_float(s[c][0]), __uint_as_float(s[c][1]));
#pragma unroll
          for (int i = 2; i < 32; i += 2) mx[c] = max3(mx[c], __uint_as_float(s[c][i]), __uint_as_float(s[c][i + 1]));
        }
        const float m_tile = max3(fmaxf(mx[0], mx[1]), mx[2], mx[3]) * sc;     // sc > 0, so the max commutes with it
        const bool raise = m_tile > m_run + kLazyMax;         // also true for the first finite maximum
        const float m_new = raise ? m_tile : m_run;
        const float m_use = m_new == -INFINITY ? 0.f : m_new;
        if (j > 0 && __any_sync(0xffffffffu, raise)) {
          // (S of this tile was computed after the stream's previous P V product: O is stable)
          const float alpha = fast_exp2(m_run - m_use);       // 1 for rows that keep their maximum
          l_run *= alpha;
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            tmem_ld32(to + 32 * c, o);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
            tmem_st32(to + 32 * c, o);
          }
          tmem_st_wait();
        }
        m_run = m_new;
        // P = exp2(S * scale - m) as bf16 over the first half of S: key pairs (2c, 2c+1) in column c.  One pair in
        // kPolyOf is a cubic on the FMA pipe (the special-function unit alone would need as long
        // as the tensor cores).
        const F2 sc2 = f2(sc, sc), m2 = f2(-m_use, -m_use);
        F2 sum[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t pw[32];
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const int i = 2 * c;
            const F2 x = fma2(f2(__uint_as_float(s[2 * h + (i >> 5)][i & 31]), __uint_as_float(s[2 * h + (i >> 5)][(i & 31) + 1])), sc2, m2);
            F2 e;
            if (c % kPolyOf == kPolyOf - 1) {
              e = poly_exp2(x);
            } else {
              const float2 y = unpack(x);
              e = f2(fast_exp2(y.x), fast_exp2(y.y));
            }
            sum[c & 1] = add2(sum[c & 1], e);
            const float2 pp = unpack(e);
            pw[c] = pack_bf16(pp.x, pp.y);
          }
          tmem_st32(ts + 32 * h, pw);
          tmem_st_wait();
          if (h == 0) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p(stream, 0));
          }
        }
        const float2 total = unpack(add2(sum[0], sum[1]));
        l_run += total.x + total.y;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (warp_idle) mbar_arrive(bar_p(stream, 0));
        mbar_arrive(bar_p(stream, 1));
      }
    }
    if (n_mine > 0) {
      ok = ok && mbar_wait(bar_o(stream), 0, fail);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
    }
    if (!two && stream == 1) s_pair[row_local] = make_float2(m_run, l_run);
    if (!ok) s_fail = 1;
    __syncwarp();
    asm volatile("setmaxnreg.dec.sync.aligned.u32 168;");
    asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool ok = s_fail == 0;
  if (!ok && tid == 0) flag_status(p.dev_status, b, TWIG_DEV_INTERNAL);
  // this thread's row: (m, l), and 32 columns of its O at a time (with the same rows in both streams, stream 0's
  // threads add up the two)
  const bool row_active = warp < 8 && (two || stream == 0);
  const bool have_o = row_active && n_my > 0 && ok && row0 + (row_local & ~31) < rows_total;     // warp-uniform
  float a0 = 1.f, a1 = 0.f;
  if (!two && have_o) {
    const float2 other = s_pair[row_local];
    const float m = fmaxf(m_run, other.x);
    a0 = l_run > 0.f ? fast_exp2(m_run - m) : 0.f;
    a1 = other.y > 0.f ? fast_exp2(other.x - m) : 0.f;
    l_run = l_run * a0 + other.y * a1;
    m_run = m;
  }
  auto load_o = [&](int ch, float (&v)[32]) {
    uint32_t x[32];
    tmem_ld32(t_lane + 256 + (two ? stream * 128 : 0) + ch * 32, x);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(x[i]);
    if (!two && n_my > 1) {
      tmem_ld32(t_lane + 384 + ch * 32, x);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = fmaf(__uint_as_float(x[i]), a1, v[i] * a0);
    }
  };
  auto release = [&]() {                           // every tensor-memory load of this CTA is done
    tc_fence_before();
    __syncthreads();
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  };

  if (n_splits == 1) {
    if (have_o) {
      const int node = row_valid ? gr / p.group : 0, h = hk * p.group + (row_valid ? gr - node * p.group : 0);
      __nv_bfloat16 *dst = p.out + (((long long)b * p.t_max + node) * p.n_q_heads + h) * kD;
      const float inv = 1.f / l_run;
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        float v[32];
        load_o(ch, v);
        if (row_valid) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint4 w;
            w.x = pack_bf16(v[8 * c] * inv, v[8 * c + 1] * inv);
            w.y = pack_bf16(v[8 * c + 2] * inv, v[8 * c + 3] * inv);
            w.z = pack_bf16(v[8 * c + 4] * inv, v[8 * c + 5] * inv);
            w.w = pack_bf16(v[8 * c + 6] * inv, v[8 * c + 7] * inv);
            st_16(dst + ch * 32 + 8 * c, w);
          }
        }
      }
      if (p.lse && row_valid) p.lse[((long long)b * p.n_q_heads + h) * p.t_max + node] = (m_run + log2f(l_run)) * 0.6931471805599453f;
    }
    release();
    return;
  }

  // ---- merge the key splits of the cluster ----
  // Once all CTAs have left their key loops every thread sends its row's (m, l) and O / l as scaled fp16 (see
  // row_scale: finer than the bf16 output whatever the magnitude of V) to the row's owner: asynchronous stores
  // that the owner's barrier counts, plain stores for the CTA's own share.
  const int rows_per = (two ? kRows : 128) / n_splits;
  unsigned char *recv = smem + 2 * kQBytes;                   // [sender * rows_per + owned row][128] fp16, in the ring
  float4 *r_ml = reinterpret_cast<float4 *>(smem);            // (m, l, row scale, -), in Q's place
  if (tid == 0) mbar_arrive_expect_tx(bar_recv, (uint32_t)((n_splits - 1) * rows_per * (kD * 2 + 16)));
  // this CTA has left its key loop; the rows' scales are found while the others leave theirs
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  float amax = 0.f;
  if (have_o) {
#pragma unroll 1
    for (int ch = 0; ch < 4; ++ch) {
      float v[32];
      load_o(ch, v);
#pragma unroll
      for (int i = 0; i < 32; ++i) amax = fmaxf(amax, fabsf(v[i]));
    }
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp < 8) {
    const int rl = row_active ? row_local : 0;
    const int owner = rl / rows_per, lr = rl % rows_per, slot = split * rows_per + lr;
    const bool remote = owner != split;
    unsigned char *ro = recv + (size_t)slot * kD * 2;
    const uint32_t ro_c = map_to_cta(smem_u32(ro), owner), bar_c = map_to_cta(bar_recv, owner);
    // (a row that saw no key in this split carries m = -inf and counts for nothing)
    const bool seen = have_o && row_valid && m_run > -INFINITY && l_run > 0.f;
    const float inv_l = seen ? 1.f / l_run : 0.f;
    float down, up;
    row_scale(seen ? amax * inv_l : 0.f, down, up);
#pragma unroll 1
    for (int ch = 0; ch < 4; ++ch) {
      float v[32];
      if (have_o) load_o(ch, v);
      if (row_active) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {              // 16-byte chunks (8 columns) are XOR-swizzled by the row to spread banks
          uint32_t h[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            h[e] = seen ? pack_f16(v[8 * i + 2 * e] * inv_l * down, v[8 * i + 2 * e + 1] * inv_l * down) : 0u;
          const int off = ((ch * 4 + i) ^ (lr & 15)) << 4;
          if (remote) st_async_b32x4(ro_c + off, h[0], h[1], h[2], h[3], bar_c);
          else *reinterpret_cast<uint4 *>(ro + off) = make_uint4(h[0], h[1], h[2], h[3]);
        }
      }
    }
    if (row_active) {
      const float mm = seen ? m_run : -INFINITY, ll = seen ? l_run : 0.f;
      if (remote) st_async_f32x4(map_to_cta(smem_u32(r_ml + slot), owner), mm, ll, up, 0.f, bar_c);
      else r_ml[slot] = make_float4(mm, ll, up, 0.f);
    }
    __syncwarp();                                  // the lanes' own-share stores come before lane 0's arrival
    if (lane == 0) mbar_arrive(bar_recv);
  }
  release();
  // (bounded by the spin limit alone: a CTA whose own key loop failed must still stay until its peers' stores
  // have landed)
  volatile int never = 0;
  const bool landed = mbar_wait(bar_recv, 0, &never);
  if (!landed) {                                   // a peer never delivered: reported, not waited for
    if (tid == 0) flag_status(p.dev_status, b, TWIG_DEV_INTERNAL);
    return;
  }
  for (int i = tid; i < rows_per * 16 && ok; i += kThreads) {           // eight columns of an owned row
    const int lr = i >> 4, c8 = i & 15, row = row0 + split * rows_per + lr;
    if (row >= rows_total) break;
    float m = -INFINITY;
    for (int sd = 0; sd < n_splits; ++sd) m = fmaxf(m, r_ml[sd * rows_per + lr].x);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float lsum = 0.f;
    for (int sd = 0; sd < n_splits; ++sd) {
      const float4 ml = r_ml[sd * rows_per + lr];
      const float wl = fast_exp2(ml.x - m) * ml.y, wgt = wl * ml.z;
      lsum += wl;
      const uint4 raw = *reinterpret_cast<const uint4 *>(recv + (size_t)(sd * rows_per + lr) * kD * 2 + ((c8 ^ (lr & 15)) << 4));
      const float2 f0 = unpack_f16(raw.x), f1 = unpack_f16(raw.y), f2 = unpack_f16(raw.z), f3 = unpack_f16(raw.w);
      acc[0] = fmaf(wgt, f0.x, acc[0]);
      acc[1] = fmaf(wgt, f0.y, acc[1]);
      acc[2] = fmaf(wgt, f1.x, acc[2]);
      acc[3] = fmaf(wgt, f1.y, acc[3]);
      acc[4] = fmaf(wgt, f2.x, acc[4]);
      acc[5] = fmaf(wgt, f2.y, acc[5]);
      acc[6] = fmaf(wgt, f3.x, acc[6]);
      acc[7] = fmaf(wgt, f3.y, acc[7]);
    }
    const float inv = 1.f / lsum;
    const int node = row / p.group, h = hk * p.group + (row - node * p.group);
    uint4 w;
    w.x = pack_bf16(acc[0] * inv, acc[1] * inv);
    w.y = pack_bf16(acc[2] * inv, acc[3] * inv);
    w.z = pack_bf16(acc[4] * inv, acc[5] * inv);
    w.w = pack_bf16(acc[6] * inv, acc[7] * inv);
    st_16(p.out + (((long long)b * p.t_max + node) * p.n_q_heads + h) * kD + c8 * 8, w);
    if (p.lse && c8 == 0)
      p.lse[((long long)b * p.n_q_heads + h) * p.t_max + node] = (m + log2f(lsum)) * 0.6931471805599453f;
  }
}

}  // namespace

// tcgen05 path: rows <= 64 transposed (tree_attn_narrow.cu), more here
twig_status launch_tree_attn_tcgen05(AttnParams &p, int batch, int rows, cudaStream_t st) {
  if (rows <= 64) return launch_tree_attn_narrow(p, batch, rows, st);
  p.row_blocks = (rows + kRows - 1) / kRows;
  if ((long long)p.n_kv_heads * p.row_blocks > 65535) return TWIG_ERR_UNSUPPORTED;
  TileMaps maps;
  if (!tile_maps(p, &maps)) return TWIG_ERR_UNSUPPORTED;
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(tree_attn_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess)
      return TWIG_ERR_CUDA;
    attr_set = true;
  }
  const int max_tiles = (p.max_len + p.t_max + kKeys - 1) / kKeys;
  int n_splits = pick_splits(batch * p.n_kv_heads * p.row_blocks, max_tiles, 1, p.forced_splits);
  // A merge costs 3 us, a tile 1.6 us with different rows in the streams and 0.85 with alternate tiles: halving a
  // short item does not pay (240 rows, 64 pairs, 3 tiles: 14.1 us whole, 15.6 halved; 72 rows, 9 tiles: 13.8, 14.0).
  if (p.forced_splits == 0 && (rows > 128 ? n_splits == 2 && max_tiles < 4 : max_tiles < (n_splits == 2 ? 8 : 4))) n_splits = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_splits, p.n_kv_heads * p.row_blocks, batch);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n_splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.overlap ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, tree_attn_wide_kernel, p, maps) == cudaSuccess ? TWIG_OK : TWIG_ERR_CUDA;
}

}  // namespace twig
