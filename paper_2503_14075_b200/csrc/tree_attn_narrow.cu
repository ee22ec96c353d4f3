// Tree attention for up to 64 query rows per kv head on the 5th-generation tensor cores, with both
// products transposed: S^T = K Q^T and O^T = V^T P^T.
//
// What bounds it is the K / V stream, so everything else has to stay out of its way.  With the keys
// (S^T) and the head dimension (O^T) on the M side of the instruction and the query rows on the N
// side, a tile of 128 keys fills all 128 lanes whatever the number of rows, where 16 to 64 rows on
// the M side used half of the lanes, half of the instruction and 256 tensor-memory columns:
//   * the chain of one tile (product, softmax, product) is paid once per 64 KB of K and V instead of
//     once per 32 KB, and takes half as long (16 or 32 elements per thread);
//   * a row is a column of S^T, so the running maximum is only looked at ("does any logit exceed
//     the reference by more than 2^8?") and never reduced, except for the first tile of an item
//     and the rare tile that raises it; row sums stay in registers until the end.
//
// head_dim 64: a tile is one panel (16 KB for K, 16 KB for V) and O^T has M = 64, 16 rows in each quadrant's first lanes.
// Half the bytes a tile, the same chain, so this one is bound by the chain and wants more CTAs (256 pairs of 64 rows
// at 1000 keys: 20.9 us a layer, 3.5 TB/s; the mma.sync kernel took 29.3).
//
// Warps 0-7 (softmax): warp w reads lanes 32 (w % 4) .. + 31 (one key per thread) and half w / 4 of
//   the rows; they also load Q.  P^T goes to shared memory as it lies in the registers: a key's
//   probabilities are contiguous (the instruction's MN-major B operand).
// Warp 8 (loader): K and V tiles (units K0 K1 V0 K2 V1 ...) into a ring of SLOTS slots by TMA;
//   the tile with the prefix end and the tree's rows by boxes of 32 and 8 rows, spread over the lanes (by
//   16-byte cp.async this tile cost one warp 1.3 us to issue); rows of V that must not count are cleared.
// Warp 9 (issuer): one elected lane issues S^T two tiles ahead and O^T += V^T P^T in order.
// Key splits of a cluster are merged through distributed shared memory: each CTA stages its O in fp32,
// sends the rows to their owners by bulk copies, and the owner adds up.
// Every wait is bounded: if one runs out the request is flagged TWIG_DEV_INTERNAL.
#include <cooperative_groups.h>
#include <cuda.h>

#include <type_traits>

#include "attn_tiles.cuh"
#include "columns.cuh"

namespace cg = cooperative_groups;

namespace twig {

namespace {

constexpr int kKeys = kTileKeys;                  // keys per tile
constexpr int kThreads = 320;
constexpr int kSoftWarps = 8;
constexpr float kLazyMax = 8.f;                    // raise a row's reference only beyond this (log2 units)

template <int D, int R, int SLOTS_, int MIN_CTAS>
struct NarrowCfg {
  static constexpr int SLOTS = SLOTS_;
  static constexpr int TILE_BYTES = tile_bytes<D>();
  static constexpr int RH = R / 2;                 // rows per softmax thread
  static constexpr int Q_BYTES = R * D * 2;        // 64-column panels of R x 128 B
  static constexpr int P_ROW = R * 2;              // bytes of a key's probabilities
  // A product of eight instructions takes 800 cycles from its issue to the barrier that reports it, as
  // long as the softmax of a tile: with one P buffer the two alternate.  Two CTAs on an SM fill each
  // other's gaps and need the shared memory for the ring; a CTA alone gets two buffers.
  static constexpr int P_BUFS = MIN_CTAS == 1 ? 2 : 1;
  static constexpr int P_ONE = kKeys * P_ROW;
  static constexpr int P_BYTES = P_BUFS * P_ONE;
  // units requested before the predecessor is waited for; the rest of the ring queues up behind Q, not in
  // front of it (Q took 3.4 us behind 192 KB per SM)
  static constexpr int PRE_UNITS = 256 / D;
  static constexpr int RING_BYTES = SLOTS * TILE_BYTES;
  static constexpr int SMEM_BYTES = Q_BYTES + P_BYTES + RING_BYTES;
  static constexpr uint32_t TMEM_COLS = R == 64 ? 256 : R == 32 ? 128 : 64;     // S^T twice, O^T: 3 R columns
  static constexpr uint32_t O_COL = 2 * R;
  // P^T is MN-major with rows of P_ROW bytes: the swizzle of that width
  static constexpr int P_LAYOUT = R == 64 ? 2 : R == 32 ? 4 : 6;
  static_assert(PRE_UNITS <= SLOTS && 2 * R * D * 4 <= RING_BYTES, "the split merge stages and receives fp32 rows in the ring");
};

// shared-memory matrix descriptor with a choice of swizzle (2: 128 B, 4: 64 B, 6: 32 B)
__device__ __forceinline__ uint64_t smem_desc_of(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t layout) {
  return (uint64_t)((addr & 0x3ffff) >> 4) | (uint64_t)((lbo >> 4) & 0x3fff) << 16 | (uint64_t)((sbo >> 4) & 0x3fff) << 32 |
         (uint64_t)1 << 46 | (uint64_t)layout << 61;
}

// bytes of this CTA's shared memory -> a cluster CTA's, counted on that CTA's barrier
__device__ __forceinline__ void bulk_to_cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "r"(src), "r"(bytes), "r"(bar) : "memory");
}

template <int D, int R, int SLOTS, int MIN_CTAS>
__global__ void __launch_bounds__(kThreads, MIN_CTAS)
tree_attn_narrow_kernel(const AttnParams p, const __grid_constant__ TileMaps maps) {
  using C = NarrowCfg<D, R, SLOTS, MIN_CTAS>;
  using RowBits = typename std::conditional<R == 64, unsigned long long, unsigned int>::type;
  constexpr int RH = C::RH, CPR = D / 8;           // 16-byte chunks of a row
  extern __shared__ __align__(1024) unsigned char smem[];
  // (static shared memory stays below 1 KB: two CTAs of the largest ring fill an SM exactly)
  __shared__ RowBits s_vis[TWIG_MAX_NODES];        // bit r of entry j: row r of this CTA sees tree node j
  __shared__ __align__(16) float s_red[4 * R];     // parents (set-up); per-quadrant column maxima / sums
  __shared__ __align__(16) float s_m[R];           // reference of every row (scaled logits, log2 units)
  __shared__ __align__(8) unsigned long long s_bar[2 * SLOTS + 9];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;

  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);     // (uniform for the compiler too: see umma8_kk)
  const int split = blockIdx.x, n_splits = gridDim.x;
  const int hk = blockIdx.y / p.row_blocks, rb = blockIdx.y % p.row_blocks;
  const int b = blockIdx.z;

  const uint32_t q_s = smem_u32(smem);
  const uint32_t p_s = q_s + C::Q_BYTES;
  const uint32_t ring_s = p_s + C::P_BYTES;
  const uint32_t bars = smem_u32(s_bar);
  auto bar_full = [&](int slot) { return bars + 8 * slot; };
  auto bar_empty = [&](int slot) { return bars + 8 * (SLOTS + slot); };
  auto bar_s = [&](int buf) { return bars + 8 * (2 * SLOTS + buf); };
  auto bar_p = [&](int buf) { return bars + 8 * (2 * SLOTS + 2 + buf); };
  auto bar_o = [&](int buf) { return bars + 8 * (2 * SLOTS + 4 + buf); };
  const uint32_t bar_q = bars + 8 * (2 * SLOTS + 6), bar_recv = bars + 8 * (2 * SLOTS + 7), bar_raw = bars + 8 * (2 * SLOTS + 8);
  const int rows_per = R / n_splits;               // rows a CTA of the cluster owns in the merge

  // ---- what needs nothing from global memory ----
  if (tid == 0) {
    s_fail = 0;
    for (int i = 0; i < SLOTS; ++i) {
      mbar_init(bar_full(i), 32);                  // every loader lane arrives once per unit
      mbar_init(bar_empty(i), 1);                  // one tcgen05.commit
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_s(i), 1);
      mbar_init(bar_p(i), kSoftWarps);
      mbar_init(bar_o(i), 1);
    }
    mbar_init(bar_q, kSoftWarps);
    mbar_init(bar_recv, 1);
    mbar_init(bar_raw, 1);
    if (n_splits > 1)                              // every peer's O rows and (m, l)
      mbar_arrive_expect_tx(bar_recv, (uint32_t)((n_splits - 1) * rows_per * (D * 4 + 16)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(C::TMEM_COLS) : "memory");
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
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(C::TMEM_COLS) : "memory");
  };

  // With `early_prefix` the lengths, the parents and the cached prefix may be read while the preceding
  // kernel drains; q, the tree's rows and the output only after it has completed.
  if (!p.early_prefix) wait_predecessor();
  const int n = p.n_nodes[b], L = p.kv_len[b];
  const int my_parent = tid < p.t_max ? p.parent[(long long)b * p.t_max + tid] : -1;
  const bool first = split == 0 && blockIdx.y == 0 && tid == 0;
  const int rows_total = n * p.group, row0 = rb * R;
  if (n <= 0 || n > p.t_max || L < 0 || L > p.max_len || row0 >= rows_total) {
    if (first && (n < 0 || n > p.t_max)) flag_status(p.dev_status, b, TWIG_DEV_BAD_TREE);
    else if (first && n > 0 && (L < 0 || L > p.max_len)) flag_status(p.dev_status, b, TWIG_DEV_OVERFLOW);
    leave();
    return;
  }
  // key positions: prefix rows 0 .. L-1, tree node j at L8 + j (whole boxes of eight rows; the gap is masked)
  const int L8 = (L + 7) & ~7, NK = L8 + n;
  const int n_tiles = (NK + kKeys - 1) / kKeys;
  const int per = (n_tiles + n_splits - 1) / n_splits;
  const int t_begin = min(n_tiles, split * per);
  const int n_my = min(n_tiles, t_begin + per) - t_begin;

  int *s_par = reinterpret_cast<int *>(s_red);
  if (tid < TWIG_MAX_NODES) s_vis[tid] = 0;
  bool bad = false;
  if (tid < n) {
    s_par[tid] = my_parent;
    bad = (tid == 0) ? (my_parent != -1) : (my_parent < 0 || my_parent >= tid);
  }
  if (__syncthreads_or(bad)) {                     // (also: barriers and the zeroed table are visible)
    if (first) flag_status(p.dev_status, b, TWIG_DEV_BAD_TREE);
    leave();
    return;
  }

  // ---- loader: unit u is K of the first tile, then K(t) and V(t-1) in turn, V of the last tile ----
  const int n_units = 2 * n_my;
  auto unit_is_v = [&](int u) { return u > 0 && (!(u & 1) || u == n_units - 1); };
  auto unit_tile = [&](int u) { return t_begin + (u == n_units - 1 ? n_my - 1 : (u & 1) ? (u + 1) >> 1 : u == 0 ? 0 : (u >> 1) - 1); };
  auto unit_in_prefix = [&](int u) { return unit_tile(u) * kKeys + kKeys <= L; };
  const TileSource source{L, L8, NK, hk, b, p.layer, b * p.n_kv_heads + hk};
  auto load_whole = [&](int u) {
    const int slot = u % SLOTS;
    load_whole_tile<D>(maps, source, unit_is_v(u), ring_s + slot * C::TILE_BYTES, bar_full(slot), unit_tile(u) * kKeys, lane);
  };
  const int n_first = min(n_units, C::PRE_UNITS);
  if (warp == 8)
    for (int u = 0; u < n_first; ++u)
      if (unit_in_prefix(u)) load_whole(u);

  // (the loader needs neither the tensor memory nor anything that is set up from here on)
  tc_fence_before();
  if (warp != 8) bar_sync(4, kThreads - 32);
  tc_fence_after();
  // (only now, with this CTA's tensor memory allocated, may CTAs of the next kernel be scheduled: they
  // could take the columns and then wait for this kernel to complete)
  wait_predecessor();
  if (warp != 8) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem = s_tmem;
  volatile int *fail = &s_fail;
  const int quad = warp & 3, half = (warp >> 2) & 1, h0 = half * RH;
  const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
  float l[RH];                                     // softmax threads: the rows' sums over this thread's keys

  if (warp == 8) {
    // ================= loader =================
    uint32_t raw_phase = 0;
    bool ok = true;
    for (int u = 0; u < n_units && ok; ++u) {
      if (u < n_first && unit_in_prefix(u)) continue;      // requested above
      if (u >= SLOTS) {
        ok = mbar_wait(bar_empty(u % SLOTS), (u / SLOTS - 1) & 1, fail);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
      }
      if (unit_in_prefix(u)) {
        load_whole(u);
      } else {
        ok = load_edge_tile<D>(maps, source, unit_is_v(u), ring_s + u % SLOTS * C::TILE_BYTES, bar_full(u % SLOTS), bar_raw, raw_phase,
                            unit_tile(u) * kKeys, lane, fail);
        ok = __all_sync(0xffffffffu, ok);
      }
    }
    if (!ok) s_fail = 1;
  } else if (warp == 9) {
    // ================= MMA issuer (one elected lane; the warp stays together) =================
    {
      const uint32_t leader = elect_one();
      // S^T: A = K (K-major), B = Q (K-major); O^T: A = V (MN-major), B = P^T (MN-major)
      constexpr uint32_t kIdescS = instr_desc(128, R, false), kIdescO = instr_desc(D, R, true) | (1u << 15);
      bool ok = true;
      auto wait_full = [&](int u) {
        if (ok) ok = mbar_wait(bar_full(u % SLOTS), (u / SLOTS) & 1, fail);
      };
      auto issue_s = [&](int it) {
        const int u = it == 0 ? 0 : 2 * it - 1;
        wait_full(u);
        if (!ok) return;
        const uint64_t kd = smem_desc(ring_s + (u % SLOTS) * C::TILE_BYTES, 16), qd = smem_desc(q_s, 16);
        if constexpr (D == 128) umma8_kk<kPanelBytes, R * 128>(leader, tmem + (it & 1) * R, kd, qd, kIdescS);
        else umma4_kk(leader, tmem + (it & 1) * R, kd, qd, kIdescS);
        umma_commit_if(leader, bar_s(it & 1));
        umma_commit_if(leader, bar_empty(u % SLOTS));
      };
      if (n_my > 0) {
        ok = mbar_wait(bar_q, 0, fail);
        issue_s(0);
      }
      if (n_my > 1) issue_s(1);
      for (int it = 0; it < n_my && ok; ++it) {
        const int u = it == n_my - 1 ? n_units - 1 : 2 * it + 2;
        ok = mbar_wait(bar_p(it & 1), (it >> 1) & 1, fail);       // P(it) is in shared memory, S(it) has been read
        wait_full(u);
        if (!ok) break;
        tc_fence_after();
        const uint64_t vd = smem_desc(ring_s + (u % SLOTS) * C::TILE_BYTES, kPanelBytes);
        const uint64_t pd = smem_desc_of(p_s + it % C::P_BUFS * C::P_ONE, 16, 8 * C::P_ROW, C::P_LAYOUT);
        const int steps = (min(kKeys, NK - (t_begin + it) * kKeys) + 15) >> 4;     // 16 keys each
        if (steps == kKeys / 16) umma8_ss<2048, 16 * C::P_ROW>(leader, tmem + C::O_COL, vd, pd, kIdescO, it > 0);
        else
          for (int j = 0; j < steps; ++j)
            if (leader) umma(tmem + C::O_COL, vd + j * 128, pd + j * C::P_ROW, kIdescO, (it > 0) || (j > 0));
        umma_commit_if(leader, bar_o(it & 1));
        umma_commit_if(leader, bar_empty(u % SLOTS));
        if (it + 2 < n_my) issue_s(it + 2);
      }
      if (!ok && lane == 0) s_fail = 1;
    }
  } else {
    // ================= softmax: one key of a tile per thread, RH rows =================
    // (no wait below is followed by a break: a failed wait marks the request and the rest runs
    // through, so that the warps meet at every barrier)
    bool ok = true;
    if (n_my > 0) {                                // Q (zero rows past the request's last row)
#pragma unroll
      for (int i = 0; i < (R * CPR + 255) / 256; ++i) {
        const int r = i * (256 / CPR) + tid / CPR, c = tid % CPR;
        if (R * CPR < 256 && r >= R) break;
        const bool valid = row0 + r < rows_total;
        const int gr = valid ? row0 + r : 0, node = gr / p.group, g = gr - node * p.group;
        const __nv_bfloat16 *src = p.q + (((long long)b * p.t_max + node) * p.n_q_heads + hk * p.group + g) * D + c * 8;
        cp_async_16(q_s + (c >> 3) * R * 128 + r * 128 + (((c & 7) ^ (r & 7)) << 4), src, valid);
      }
      cp_async_commit();
    }
    // meanwhile: which rows see which tree node (node i's rows see i and its ancestors; s_par and s_red share
    // their memory, so nobody goes on before everybody is done)
    if (tid < n) {
      const int lo = max(tid * p.group - row0, 0), hi = min((tid + 1) * p.group - row0, R);
      if (hi > lo) {
        // (32-bit words: a 64-bit atomicOr in shared memory is a compare-and-swap loop, and every node meets
        // every other one at the root)
        const unsigned long long rows = (hi == 64 ? ~0ull : (1ull << hi) - 1ull) & ~((1ull << lo) - 1ull);
        for (int x = tid; x >= 0; x = s_par[x]) {
          unsigned int *word = reinterpret_cast<unsigned int *>(s_vis + x);
          if ((unsigned int)rows) atomicOr(word, (unsigned int)rows);
          if (R == 64 && (unsigned int)(rows >> 32)) atomicOr(word + 1, (unsigned int)(rows >> 32));
        }
      }
    }
    if (n_my > 0) {
      cp_async_wait<0>();
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_q);
    }
    bar_sync(3, 32 * kSoftWarps);
#pragma unroll
    for (int i = 0; i < RH; ++i) l[i] = 0.f;
    const int kl = quad * 32 + lane;               // this thread's key within a tile
    const float sc = p.scale_log2;
    for (int it = 0; it < n_my; ++it) {
      const int vj = (t_begin + it) * kKeys + kl;
      const bool edge = (t_begin + it) * kKeys + kKeys > L;      // (uniform) some keys are not in the prefix
      RowBits vis = ~(RowBits)0;                   // this key's rows; bit i: row h0 + i
      if (edge && vj >= L) vis = vj >= L8 && vj < NK ? s_vis[vj - L8] >> h0 : 0;
      ok = ok && mbar_wait(bar_s(it & 1), (it >> 1) & 1, fail);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      const uint32_t ts = t_lane + (it & 1) * R + h0;
      uint32_t sr[RH];
      auto subtract_references = [&]() {           // scaled logits minus the rows' references
#pragma unroll
        for (int i = 0; i < RH; i += 4) {
          const float4 m = *reinterpret_cast<const float4 *>(s_m + h0 + i);
          sr[i] = __float_as_uint(fmaf(__uint_as_float(sr[i]), sc, -m.x));
          sr[i + 1] = __float_as_uint(fmaf(__uint_as_float(sr[i + 1]), sc, -m.y));
          sr[i + 2] = __float_as_uint(fmaf(__uint_as_float(sr[i + 2]), sc, -m.z));
          sr[i + 3] = __float_as_uint(fmaf(__uint_as_float(sr[i + 3]), sc, -m.w));
        }
        if (edge)
#pragma unroll
          for (int i = 0; i < RH; ++i)
            if (!((vis >> i) & 1)) sr[i] = 0xff800000u;          // -inf
      };
      auto wait_o = [&](int i) {                   // P(i) V(i) has completed
        ok = ok && mbar_wait(bar_o(i & 1), (i >> 1) & 1, fail);
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
      };
      tmem_load<RH>(ts, sr);
      bool fresh = it == 0, raise = true;          // fresh: the rows have no reference yet
      if (fresh && !edge) {
        // A first reference that needs no reduction: the largest logit of four of the tile's keys, position 0
        // among them (where models put an attention sink).  It only has to lie less than 2^8 below the
        // row's maximum, which is checked like any other tile's.
        if (lane == 0)
#pragma unroll
          for (int i = 0; i < RH; i += 4)
            *reinterpret_cast<uint4 *>(s_red + quad * R + h0 + i) = make_uint4(sr[i], sr[i + 1], sr[i + 2], sr[i + 3]);
        bar_sync(1 + half, 128);
        if (quad == 0 && lane < RH) {
          const int r = h0 + lane;
          s_m[r] = sc * fmaxf(fmaxf(s_red[r], s_red[R + r]), fmaxf(s_red[2 * R + r], s_red[3 * R + r]));
        }
        bar_sync(1 + half, 128);
        fresh = false;
      }
      if (!fresh) {
        subtract_references();
        float mx = -INFINITY;
#pragma unroll
        for (int i = 0; i < RH; ++i) mx = fmaxf(mx, __uint_as_float(sr[i]));
        raise = bar_any(1 + half, 128, mx > kLazyMax);
      }
      if (raise) {
        // new references: column maxima over the warp's keys, over the four warps of this half, then
        // the rows' sums and O are rescaled
        float mine = -INFINITY;                    // lane i: the warp's maximum of row h0 + i
        tmem_load<RH>(ts, sr);
#pragma unroll
        for (int i = 0; i < RH; ++i) {
          const float mx = warp_max(((vis >> i) & 1) ? __uint_as_float(sr[i]) * sc : -INFINITY);
          if (lane == i) mine = mx;
        }
        if (lane < RH) s_red[quad * R + h0 + lane] = mine;
        bar_sync(1 + half, 128);
        if (quad == 0 && lane < RH) {
          const int r = h0 + lane;
          const float mx = fmaxf(fmaxf(s_red[r], s_red[R + r]), fmaxf(s_red[2 * R + r], s_red[3 * R + r]));
          // (a row that sees no key of the first tile keeps the reference 0: that tile is then the last one)
          const float old = fresh ? 0.f : s_m[r];
          const bool up = mx > -INFINITY && (fresh || mx > old + kLazyMax);
          s_m[r] = up ? mx : old;
          s_red[r] = up ? fast_exp2(old - mx) : 1.f;
        }
        bar_sync(1 + half, 128);
        if (it > 0) {
          wait_o(it - 1);                          // O is stable
          uint32_t o[RH];
          tmem_load<RH>(t_lane + C::O_COL + h0, o);
#pragma unroll
          for (int i = 0; i < RH; ++i) {
            const float a = s_red[h0 + i];
            l[i] *= a;
            o[i] = __float_as_uint(__uint_as_float(o[i]) * a);
          }
          tmem_store<RH>(t_lane + C::O_COL + h0, o);
        }
        tmem_load<RH>(ts, sr);
        subtract_references();
      }
      // P^T = exp2(..) as bf16: this key's rows are contiguous, 16-byte chunks XORed with the swizzle
      uint32_t pw[RH / 2];
      auto exps = [&](int i) {
        const float p0 = fast_exp2(__uint_as_float(sr[i])), p1 = fast_exp2(__uint_as_float(sr[i + 1]));
        l[i] += p0;
        l[i + 1] += p1;
        pw[i / 2] = pack_bf16(p0, p1);
      };
#pragma unroll
      for (int i = 0; i < RH; i += 2) exps(i);
      if (it >= C::P_BUFS) wait_o(it - C::P_BUFS);           // this P buffer is free
      const uint32_t prow = p_s + it % C::P_BUFS * C::P_ONE + kl * C::P_ROW, swz = ((kl * C::P_ROW) >> 7) & (C::P_ROW / 16 - 1);
#pragma unroll
      for (int k = 0; k < RH / 8; ++k)
        asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(prow + (((h0 / 8 + k) ^ swz) << 4)), "r"(pw[4 * k]),
                     "r"(pw[4 * k + 1]), "r"(pw[4 * k + 2]), "r"(pw[4 * k + 3]) : "memory");
      fence_async_smem();                          // P was written with ordinary stores
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p(it & 1));
    }
    if (n_my > 0) {
      ok = ok && mbar_wait(bar_o((n_my - 1) & 1), ((n_my - 1) >> 1) & 1, fail);      // the last product has completed
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
    }
    if (!ok) s_fail = 1;
    // row sums over the warp's keys
    const float sum = column_reduce<RH>(l, lane, [](float x, float y) { return x + y; });
    bar_sync(1 + half, 128);                       // (the maxima in s_red have been read)
    if ((lane & (32 / RH - 1)) == 0) s_red[quad * R + h0 + lane / (32 / RH)] = sum;
  }
  __syncwarp();
  // every unit that was requested has been used, every product has completed: the ring is free
  if (n_splits > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  float *stage = reinterpret_cast<float *>(smem + C::Q_BYTES + C::P_BYTES);     // [row][D] fp32
  if (warp < kSoftWarps) {
    uint32_t o[RH];
    if (n_my > 0) tmem_load<RH>(t_lane + C::O_COL + h0, o);
#pragma unroll
    for (int i = 0; i < RH; ++i)                   // (64 rows of O^T: 16 in each quadrant's first lanes)
      if (D == 128 || lane < 16) stage[(h0 + i) * D + quad * (D / 4) + lane] = n_my > 0 ? __uint_as_float(o[i]) : 0.f;
    if (n_splits > 1) fence_async_smem();          // (the rows leave by bulk copies)
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
  const bool ok = s_fail == 0;
  if (!ok && tid == 0) flag_status(p.dev_status, b, TWIG_DEV_INTERNAL);
  auto row_sum = [&](int r) { return n_my > 0 ? (s_red[r] + s_red[R + r]) + (s_red[2 * R + r] + s_red[3 * R + r]) : 0.f; };
  // eight columns of one row (a row is D / 8 consecutive threads), and its log-sum-exp
  auto store_row8 = [&](int r, int c, const float (&acc)[8], float lsum, float m) {
    const int gr = row0 + r, node = p.group == 1 ? gr : gr / p.group, h = hk * p.group + (gr - node * p.group);
    const float inv = 1.f / lsum;
    uint4 packed;
    packed.x = pack_bf16(acc[0] * inv, acc[1] * inv);
    packed.y = pack_bf16(acc[2] * inv, acc[3] * inv);
    packed.z = pack_bf16(acc[4] * inv, acc[5] * inv);
    packed.w = pack_bf16(acc[6] * inv, acc[7] * inv);
    st_16(p.out + (((long long)b * p.t_max + node) * p.n_q_heads + h) * D + c, packed);
    if (p.lse && c == 0)
      p.lse[((long long)b * p.n_q_heads + h) * p.t_max + node] = (m + log2f(lsum)) * 0.6931471805599453f;
  };
  const int n_rows = min(R, rows_total - row0);
  if (n_splits == 1) {
    if (ok) {
#pragma unroll
      for (int k = 0; k < (R * CPR + kThreads - 1) / kThreads; ++k) {
        const int i = tid + k * kThreads, r = i / CPR, c = i % CPR * 8;
        if (r < n_rows) {
          float acc[8];
          *reinterpret_cast<float4 *>(acc) = *reinterpret_cast<const float4 *>(stage + r * D + c);
          *reinterpret_cast<float4 *>(acc + 4) = *reinterpret_cast<const float4 *>(stage + r * D + c + 4);
          store_row8(r, c, acc, row_sum(r), s_m[r]);
        }
      }
    }
    return;
  }

  // ---- merge the key splits of the cluster: every CTA owns R / n_splits rows ----
  // received O rows: [sender][owned row][D] fp32 behind the stage; (m, l): [sender][owned row] in P's place
  float *recv = stage + R * D;
  float4 *recv_ml = reinterpret_cast<float4 *>(smem + C::Q_BYTES);
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // every peer has left its key loop
  if (warp == 0 && lane < n_splits && lane != split) {                    // one copy per owner
    const uint32_t dst = map_to_cta(smem_u32(recv + (size_t)split * rows_per * D), lane);
    bulk_to_cluster(dst, smem_u32(stage + (size_t)lane * rows_per * D), (uint32_t)(rows_per * D * 4), map_to_cta(bar_recv, lane));
  }
  if (tid >= 32 && tid < 32 + R) {
    const int r = tid - 32, owner = r / rows_per;
    const float lr = row_sum(r), mr = lr > 0.f ? s_m[r] : -INFINITY;      // (saw no key in this split: counts for nothing)
    float4 *dst = recv_ml + split * rows_per + (r - owner * rows_per);
    if (owner == split) *dst = make_float4(mr, lr, 0.f, 0.f);
    else st_async_f32x4(map_to_cta(smem_u32(dst), owner), mr, lr, 0.f, 0.f, map_to_cta(bar_recv, owner));
  }
  __syncthreads();
  const bool landed = mbar_wait(bar_recv, 0, fail);
  if (!landed && tid == 0) flag_status(p.dev_status, b, TWIG_DEV_INTERNAL);
  if (landed && ok)
    for (int i = tid; i < rows_per * CPR; i += kThreads) {
      const int lr = i / CPR, c = i % CPR * 8;
      if (split * rows_per + lr >= n_rows) break;
      float m = -INFINITY;
      for (int s = 0; s < n_splits; ++s) m = fmaxf(m, recv_ml[s * rows_per + lr].x);
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      float lsum = 0.f;
      for (int s = 0; s < n_splits; ++s) {
        const float4 ml = recv_ml[s * rows_per + lr];
        const float w = fast_exp2(ml.x - m);
        const float *src = (s == split ? stage + (size_t)(split * rows_per + lr) * D : recv + (size_t)(s * rows_per + lr) * D) + c;
        float v[8];
        *reinterpret_cast<float4 *>(v) = *reinterpret_cast<const float4 *>(src);
        *reinterpret_cast<float4 *>(v + 4) = *reinterpret_cast<const float4 *>(src + 4);
        lsum = fmaf(w, ml.y, lsum);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = fmaf(w, v[e], acc[e]);
      }
      store_row8(split * rows_per + lr, c, acc, lsum, m);
    }
  // a CTA stays until the copies out of its stage have been read
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int D, int R, int SLOTS, int MIN_CTAS>
twig_status launch_narrow(const AttnParams &p, const TileMaps &maps, int batch, int n_splits, cudaStream_t st) {
  using C = NarrowCfg<D, R, SLOTS, MIN_CTAS>;
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(tree_attn_narrow_kernel<D, R, SLOTS, MIN_CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             C::SMEM_BYTES) != cudaSuccess)
      return TWIG_ERR_CUDA;
    attr_set = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_splits, p.n_kv_heads * p.row_blocks, batch);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
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
  return cudaLaunchKernelEx(&cfg, tree_attn_narrow_kernel<D, R, SLOTS, MIN_CTAS>, p, maps) == cudaSuccess ? TWIG_OK : TWIG_ERR_CUDA;
}

}  // namespace

twig_status launch_tree_attn_narrow(AttnParams &p, int batch, int rows, cudaStream_t st) {
  p.row_blocks = 1;
  if (p.n_kv_heads > 65535) return TWIG_ERR_UNSUPPORTED;
  TileMaps maps;
  if (!tile_maps(p, &maps))
    return TWIG_ERR_UNSUPPORTED;
  // Measured on chains of layers (us per launch, 32 kv heads; T nodes at L keys):
  //   at most 148 items: one CTA per SM with a deep ring, keys split over clusters below 75 items (T = 64, B = 4,
  //     L = 1500: 22.9, with two split CTAs per SM 26.4; T = 32, B = 4, L = 250: 8.4 against 10.0). Only up to 74
  //     items of 32 rows, whose splits are short, two CTAs per SM are a little faster (B = 2, L = 1000: 11.7, 12.5).
  //   more: two CTAs per SM, whose start and end overlap (T = 64, B = 8, L = 1500: 42.2 against 48.0; T = 32,
  //     B = 16, L = 1500: 67.4 against 80.9).
  const int items = batch * p.n_kv_heads, max_tiles = (p.max_len + p.t_max + kKeys - 1) / kKeys;
  // Long caches are an exception where one CTA per SM leaves SMs idle (at most 74 CTAs with all the splits that are
  // resident at once), and with head_dim 64 always: half the bytes per tile, so the chain of a tile is what
  // more CTAs hide (T = 60, L = 8000, head_dim 128, 16 items: 26.1 and 22.7, 36 items: 46.0 and 37.5; head_dim 64, 64
  // items: 43.1 and 32.9; the other way round below 3000 keys, 16 items at 1000 keys: 10.0 and 11.0).
  const int splits1 = pick_splits(items, max_tiles, 1, p.forced_splits);
  const bool spread = p.max_len >= 3000 && (p.head_dim == 64 || items * splits1 <= 74);
  const bool single = items <= 148 && (rows > 32 || items > 74) && !spread;
  const int n_splits = single ? splits1 : pick_splits(items, max_tiles, 2, p.forced_splits);
  if (p.head_dim == 64) {
    if (rows <= 16) return single ? launch_narrow<64, 16, 10, 1>(p, maps, batch, n_splits, st) : launch_narrow<64, 16, 6, 2>(p, maps, batch, n_splits, st);
    if (rows <= 32) return single ? launch_narrow<64, 32, 10, 1>(p, maps, batch, n_splits, st) : launch_narrow<64, 32, 6, 2>(p, maps, batch, n_splits, st);
    return single ? launch_narrow<64, 64, 8, 1>(p, maps, batch, n_splits, st) : launch_narrow<64, 64, 5, 2>(p, maps, batch, n_splits, st);
  }
  if (rows <= 16) return single ? launch_narrow<128, 16, 5, 1>(p, maps, batch, n_splits, st) : launch_narrow<128, 16, 3, 2>(p, maps, batch, n_splits, st);
  if (rows <= 32) return single ? launch_narrow<128, 32, 5, 1>(p, maps, batch, n_splits, st) : launch_narrow<128, 32, 3, 2>(p, maps, batch, n_splits, st);
  return single ? launch_narrow<128, 64, 4, 1>(p, maps, batch, n_splits, st) : launch_narrow<128, 64, 2, 2>(p, maps, batch, n_splits, st);
}

}  // namespace twig
