// Draft-side token tree of tree-based self-speculative decoding (Sec. 4.3; Appendix, "Tree-based
// self-speculative decoding"): level by level, every node selected for expansion gets its E most
// probable next tokens as children; the K best nodes of a level are expanded at the next; at the end
// the tree is cut to N_max nodes.  A node's score is the log of the joint probability of its path.
// The draft model itself runs between these calls: its logits are inputs.
//
// Tree state per request (capacity `cap` nodes, node 0 = root): token, parent, score, all in
// creation order (a parent always precedes its children).
//
// A level costs one launch: the expansion kernel's CTAs of a request take a ticket when their
// children are written, and the last of them runs the step that consumes the level (the choice of the
// next level's expansion nodes, or the final pruning).  The two steps also exist as launches of
// their own.
#include "vocab_row.cuh"

namespace twig {

namespace {

constexpr int kMaxE = 16;            // children per expanded node
constexpr int kPeerStride = kMaxE + 2;   // a slice's list, its (max, sum), rows of 16 bytes
constexpr int kMaxCand = 1024;       // entries at or above the threshold that the short list holds
constexpr int kSelThreads = 256;
constexpr int kRegWords = 12;        // 32-node words of a level that one warp holds in registers

// (value, index) order of the top lists: larger value first, equal values: lower index first; and as one
// number, the larger first (-0 and 0 are equal)
__device__ __forceinline__ unsigned long long top_key(float v, int i) {
  return (unsigned long long)order_key(v + 0.f) << 32 | (0xffffffffu - (unsigned int)i);
}
__device__ __forceinline__ float top_value(unsigned long long k) {
  const uint32_t u = (uint32_t)(k >> 32);
  return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u);
}
__device__ __forceinline__ int top_index(unsigned long long k) { return (int)(0xffffffffu - (unsigned int)k); }
__device__ __forceinline__ bool comes_first(float v, int i, float w, int j) { return v > w || (v == w && i < j); }

// What follows a level: the ranking of nodes lo..hi-1 by (score desc, id asc), of which the first
// `take` are kept.
//  * expansion mode (parent_out == nullptr): their ids, ascending, to sel_out[b, 0..take) (-1 padded);
//  * final mode: the root and the selected nodes are renumbered in creation order and written as
//    parent_out / tok_out [b, t_max] with n_nodes_out[b]; kept_out[b, i] = the old id of new node i.
struct SelectArgs {
  int lo, hi, take;
  int *sel_out;
  int sel_stride;
  int *parent_out, *tok_out, *n_nodes_out, *kept_out;
  int t_max;
};

// Runs in one CTA (all of its threads) for request b.  `work` holds 2*cap words of shared memory.
// The tree state is read through L2: inside the expansion kernel the nodes of the new level were
// written by other CTAs a moment ago, and a line of this SM's L1 may predate them.
// What bounds it is latency, of memory and of cold instructions (one CTA runs this code once per launch): scores,
// parents and tokens are requested together, one warp finds the score of the last selected node bit by bit
// (a rank for every node was 100,000 comparisons at 310 nodes), and a node's position among the kept is
// counted from one bit per node.  310 nodes took 8.0 us.
__device__ void select_nodes(const SelectArgs &a, int b, int cap, const float *node_score, const int *node_tok,
                             const int *node_parent, unsigned char *work, int *dev_status) {
  uint32_t *key = reinterpret_cast<uint32_t *>(work);              // [hi], order-preserving
  unsigned int *kept_bits = key + cap;                             // [words], then the kept before each word
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int lo = a.lo, hi = a.hi, words = (hi + 31) >> 5;
  unsigned int *kept_before = kept_bits + words;
  const bool final_mode = a.parent_out != nullptr;
  const long long base = (long long)b * cap;
  const int first_parent = final_mode && tid < hi ? __ldcg(node_parent + base + tid) : -1;
  const int first_tok = final_mode && tid < hi ? __ldcg(node_tok + base + tid) : -1;
  for (int i = tid; i < hi; i += nt) key[i] = order_key(__ldcg(node_score + base + i) + 0.f);   // (-0 and 0 are equal)
  __syncthreads();
  if (tid < 32) {
    // the largest t with at least `take` keys >= t (the take-th largest key, or anything below it that as many
    // reach), from the first bit in which the keys differ; then the kept nodes, 32 to a word.  Up to
    // kRegWords words of keys stay in the lanes' registers.
    const int take = min(a.take, hi - lo), w0 = lo >> 5;
    auto run = [&](auto &&for_words) {
      uint32_t low = 0xffffffffu, high = 0;
      for_words([&](int, uint32_t k, bool in) {
        low = min(low, in ? k : 0xffffffffu);
        high = max(high, k);
      });
      low = __reduce_min_sync(0xffffffffu, low);
      high = __reduce_max_sync(0xffffffffu, high);
      uint32_t bit = low == high ? 0u : 0x80000000u >> __clz(low ^ high);
      uint32_t t = bit == 0 ? low : low & ~(2 * bit - 1);
      int reach = hi - lo;
#pragma unroll 1
      for (; bit != 0 && reach != take; bit >>= 1) {
        int c = 0;
        for_words([&](int, uint32_t k, bool) { c += k >= (t | bit) ? 1 : 0; });
        c = __reduce_add_sync(0xffffffffu, c);
        if (c >= take) {
          t |= bit;
          reach = c;
        }
      }
      // more than `take` only with equal keys at t: the lowest ids of them
      int left = 0;
      if (reach > take) {
        for_words([&](int, uint32_t k, bool) { left += k == t ? 1 : 0; });
        left = __reduce_add_sync(0xffffffffu, left) - (reach - take);
      }
      int before = 0;
      for_words([&](int w, uint32_t k, bool in) {
        bool kept = in && take > 0 && k >= t;
        if (reach > take) {
          const unsigned eqs = __ballot_sync(0xffffffffu, in && k == t);
          if (in && k == t) kept = __popc(eqs & ((1u << lane) - 1u)) < left;
          left -= __popc(eqs);
        }
        if (final_mode && 32 * w + lane == 0) kept = true;         // the root is always kept
        const unsigned bits = __ballot_sync(0xffffffffu, kept);
        if (lane == 0) {
          kept_bits[w] = bits;
          kept_before[w] = before;
        }
        before += __popc(bits);
      });
    };
    for (int w = lane; w < w0; w += 32) kept_bits[w] = kept_before[w] = 0;
    if (words - w0 <= kRegWords) {
      uint32_t k[kRegWords];
#pragma unroll
      for (int q = 0; q < kRegWords; ++q) {
        const int i = 32 * (w0 + q) + lane;
        k[q] = i >= lo && i < hi ? key[i] : 0u;                    // (no key is 0)
      }
      run([&](auto &&f) {
#pragma unroll
        for (int q = 0; q < kRegWords; ++q)
          if (w0 + q < words) f(w0 + q, k[q], k[q] != 0u);
      });
    } else {
      run([&](auto &&f) {
#pragma unroll 1
        for (int w = w0; w < words; w += kRegWords) {              // (a batch of loads in flight: with one load
          uint32_t k[kRegWords];                                   // after another 466 nodes took 13 us longer)
#pragma unroll
          for (int q = 0; q < kRegWords; ++q) {
            const int i = 32 * (w + q) + lane;
            k[q] = i >= lo && i < hi ? key[i] : 0u;
          }
#pragma unroll
          for (int q = 0; q < kRegWords; ++q)
            if (w + q < words) f(w + q, k[q], k[q] != 0u);
        }
      });
    }
  }
  __syncthreads();
  const int total = kept_before[words - 1] + __popc(kept_bits[words - 1]);
  auto position = [&](int i) {                                     // among the kept, in id order; -1: not kept
    const unsigned bits = kept_bits[i >> 5];
    return (bits >> (i & 31)) & 1u ? (int)kept_before[i >> 5] + __popc(bits & ((1u << (i & 31)) - 1u)) : -1;
  };
  const int stride = final_mode ? a.t_max : a.sel_stride;
  const long long out = (long long)b * stride;
#pragma unroll 1
  for (int k = total + tid; k < stride; k += nt) {
    if (final_mode) {
      a.parent_out[out + k] = -1;
      a.tok_out[out + k] = 0;
      if (a.kept_out) a.kept_out[out + k] = -1;
    } else {
      a.sel_out[out + k] = -1;
    }
  }
  if (final_mode && tid == 0) a.n_nodes_out[b] = total;
#pragma unroll 1
  for (int i = tid; i < hi; i += nt) {
    const int ni = position(i);
    if (ni < 0 || ni >= stride) continue;
    if (!final_mode) {
      a.sel_out[out + ni] = i;
      continue;
    }
    const int parent = i == tid ? first_parent : __ldcg(node_parent + base + i);
    const int np = i > 0 && parent >= 0 && parent < i ? position(parent) : -1;
    if (i > 0 && np < 0) flag_status(dev_status, b, TWIG_DEV_BAD_TREE);   // not a tree, or the kept set is not closed under parents
    a.parent_out[out + ni] = np;
    a.tok_out[out + ni] = i == 0 ? -1 : i == tid ? first_tok : __ldcg(node_tok + base + i);
    if (a.kept_out) a.kept_out[out + ni] = i;
  }
}

// The selection as a launch of its own: one CTA per request.
__global__ void __launch_bounds__(kSelThreads)
tree_select_kernel(const float *node_score, const int *node_tok, const int *node_parent, int cap, SelectArgs a,
                   int *dev_status) {
  extern __shared__ __align__(16) unsigned char sel_smem[];
  grid_dependency_sync();
  select_nodes(a, blockIdx.x, cap, node_score, node_tok, node_parent, sel_smem, dev_status);
}

// One cluster per (expansion slot, request), one CTA per slice of the row (see vocab_row.cuh).
// Pass 1 over the slice, eight 16-byte loads per thread in flight: running (max, sum of exp).  The E-th
// largest of the maxima of 32 groups of threads bounds the E-th largest logit of the slice from below, so
// pass 2 (over the chunks' maxima kept in registers when the slice is one batch of loads, else over the slice
// again) collects the few entries at or above it into a short list, which is ranked by counting (every candidate counts the candidates that come
// before it in the (value, index) order).  If the list overflows (e.g. a row of equal logits), E rounds run
// over the slice instead: round e finds the best entry that comes strictly after round e-1's winner, so
// nothing has to be marked as taken.  The slices' lists and sums meet in the first CTA, which ranks them the
// same way and writes the children's tokens, parents and scores.
// One CTA per row, staging it in shared memory, took 11 to 23 us a level (32000 bf16 logits, 16 x 10 rows).
struct SliceTop {
  unsigned long long *peer;    // [kMaxSlices][kPeerStride], shared: the lists (top_key; 0: no entry), (max, sum)
  uint32_t bar;
  int rank, slices;
};

template <bool FP32>
__device__ __forceinline__ void expand_row(const unsigned char *__restrict__ row, int vocab, int E, const SliceTop &st,
                                           int u, int level_base, long long base, int first, int *node_tok,
                                           int *node_parent, float *node_score, int *dev_status, int b) {
  using F = RowFormat<FP32>;
  constexpr int EPC = F::EPC;
  constexpr int kGroups = kRowThreads / 8;
  __shared__ float s_v[kRowThreads / 32];
  __shared__ int s_i[kRowThreads / 32];
  __shared__ float s_m[kRowThreads / 32], s_s[kRowThreads / 32];
  __shared__ __align__(16) float s_gmax[kGroups];
  __shared__ float s_thr;
  __shared__ unsigned long long s_cand[kMaxCand];
  __shared__ int s_n_cand;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunks = vocab / EPC, per = (chunks + st.slices - 1) / st.slices;
  const int c_first = st.rank * per, c_last = min(chunks, c_first + per);
  const bool with_tail = st.rank == 0 && chunks * EPC < vocab;     // the elements past the last whole chunk
  unsigned long long *mine = st.peer + st.rank * kPeerStride;

  // ---- pass 1 ----
  float m = -INFINITY, s = 0.f;
  auto take = [&](const float (&v)[EPC]) {
    float cm = v[0];
#pragma unroll
    for (int k = 1; k < EPC; ++k) cm = fmaxf(cm, v[k]);
    const float nm = fmaxf(m, cm);
    const float ref = nm == -INFINITY ? 0.f : nm;     // (only -inf so far: every term is exp(-inf) = 0)
    float acc = s * __expf(m - ref);
#pragma unroll
    for (int k = 0; k < EPC; ++k) acc += __expf(v[k] - ref);
    s = acc;
    m = nm;
  };
  uint4 w[kRowDeep];                                 // the slice, when it is one batch
  float cmax[kRowDeep];                              // its chunks' maxima
  const bool one_batch = c_last - c_first <= kRowDeep * kRowThreads;
  for (int c0 = c_first + tid; c0 < c_last; c0 += kRowDeep * kRowThreads) {
#pragma unroll
    for (int q = 0; q < kRowDeep; ++q)
      if (c0 + q * kRowThreads < c_last) w[q] = ld_nc_16(row + (long long)(c0 + q * kRowThreads) * 16);
    // the batch's maximum first, then one reference for its exponentials
    float bm = m;
#pragma unroll
    for (int q = 0; q < kRowDeep; ++q)
      if (c0 + q * kRowThreads < c_last) {
        float v[EPC];
        F::unpack(w[q], v);
        cmax[q] = v[0];
#pragma unroll
        for (int k = 1; k < EPC; ++k) cmax[q] = fmaxf(cmax[q], v[k]);
        bm = fmaxf(bm, cmax[q]);
      }
    const float ref = bm == -INFINITY ? 0.f : bm;
    float acc = s * __expf(m - ref), acc2 = 0.f;
#pragma unroll
    for (int q = 0; q < kRowDeep; ++q)
      if (c0 + q * kRowThreads < c_last) {
        float v[EPC];
        F::unpack(w[q], v);
#pragma unroll
        for (int k = 0; k < EPC; k += 2) {
          acc += __expf(v[k] - ref);
          acc2 += __expf(v[k + 1] - ref);
        }
      }
    s = acc + acc2;
    m = bm;
  }
  if (with_tail && tid == 0) {
    float v[EPC];
    F::tail(row, chunks, vocab, v);
    take(v);
  }
  // (the root's score is 0 by definition; its entry may be written by another CTA of this launch)
  const bool usable = u >= 0 && u < level_base;
  const float parent_score = usable && u > 0 && st.rank == 0 ? __ldcg(node_score + base + u) : 0.f;
  float g_max = m;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) g_max = fmaxf(g_max, __shfl_xor_sync(0xffffffffu, g_max, o));
  if ((lane & 7) == 0) s_gmax[tid >> 3] = g_max;
  // the warp's maximum (of its four groups), then its sum with one rescaling per lane
  g_max = fmaxf(g_max, __shfl_xor_sync(0xffffffffu, g_max, 8));
  g_max = fmaxf(g_max, __shfl_xor_sync(0xffffffffu, g_max, 16));
  if (tid == 0) s_n_cand = 0;
  __syncthreads();
  if (tid < kGroups) {                               // (one warp; the others go on to the sums)
    const float g = s_gmax[tid];
    int above = 0;                                   // group maxima ranked before mine (ties: lower group first)
#pragma unroll
    for (int j = 0; j < kGroups / 4; ++j) {
      const float4 x = reinterpret_cast<const float4 *>(s_gmax)[j];
      above += (x.x > g || (x.x == g && 4 * j < tid) ? 1 : 0) + (x.y > g || (x.y == g && 4 * j + 1 < tid) ? 1 : 0) +
               (x.z > g || (x.z == g && 4 * j + 2 < tid) ? 1 : 0) + (x.w > g || (x.w == g && 4 * j + 3 < tid) ? 1 : 0);
    }
    if (above == E - 1) s_thr = g;                   // exactly one group has this rank
  }
  s *= m == -INFINITY ? 0.f : __expf(m - g_max);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    s_m[warp] = g_max;
    s_s[warp] = s;
  }
  __syncthreads();
  const float thr = s_thr;

  // ---- pass 2: the entries at or above the threshold ----
  auto offer = [&](float v, int i) {
    if (v >= thr) {
      const int at = atomicAdd(&s_n_cand, 1);
      if (at < kMaxCand) s_cand[at] = top_key(v, i);
    }
  };
  // the chunks that hold one are found first, so that the code of an offer exists once
  auto offer_hits = [&](unsigned int hits, int c0) {
#pragma unroll 1
    for (; hits; hits &= hits - 1) {
      const int q = __ffs(hits) - 1;
      uint4 x = w[0];
#pragma unroll
      for (int i = 1; i < kRowDeep; ++i)
        if (i == q) x = w[i];
      float v[EPC];
      F::unpack(x, v);
#pragma unroll
      for (int k = 0; k < EPC; ++k) offer(v[k], (c0 + q * kRowThreads) * EPC + k);
    }
  };
  if (one_batch) {
    unsigned int hits = 0;
#pragma unroll
    for (int q = 0; q < kRowDeep; ++q)
      if (c_first + tid + q * kRowThreads < c_last && cmax[q] >= thr) hits |= 1u << q;
    offer_hits(hits, c_first + tid);
  } else {
#pragma unroll 1
    for (int c0 = c_first + tid; c0 < c_last; c0 += kRowDeep * kRowThreads) {
      unsigned int hits = 0;
#pragma unroll
      for (int q = 0; q < kRowDeep; ++q)
        if (c0 + q * kRowThreads < c_last) w[q] = *reinterpret_cast<const uint4 *>(row + (size_t)(c0 + q * kRowThreads) * 16);
#pragma unroll
      for (int q = 0; q < kRowDeep; ++q)
        if (c0 + q * kRowThreads < c_last) {
          float v[EPC];
          F::unpack(w[q], v);
          float cm = v[0];
#pragma unroll
          for (int k = 1; k < EPC; ++k) cm = fmaxf(cm, v[k]);
          if (cm >= thr) hits |= 1u << q;
        }
      offer_hits(hits, c0);
    }
  }
  if (with_tail)
    for (int i = chunks * EPC + tid; i < vocab; i += kRowThreads) offer(F::element(row, i), i);
  __syncthreads();
  const int n_cand = s_n_cand;
  const bool short_list = n_cand <= kMaxCand;

  if (short_list) {                                  // ranked by counting (indices are distinct, so ranks are)
    for (int j = tid; j < n_cand; j += kRowThreads) {
      const unsigned long long x = s_cand[j];
      int rank = 0;
#pragma unroll 4
      for (int q = 0; q < n_cand; ++q) rank += s_cand[q] > x ? 1 : 0;
      if (rank < E) mine[rank] = x;
    }
  } else {                                           // or E rounds over the whole slice
    float pv = INFINITY;                             // previous winner; every finite logit comes after (+inf, -1)
    int pi = -1;
    for (int e = 0; e < E; ++e) {
      float bv = -INFINITY;
      int bi = 0x7fffffff;
      auto best_of = [&](float v, int i) {
        const bool after_prev = pv > v || (pv == v && pi < i);
        if (after_prev && comes_first(v, i, bv, bi)) {
          bv = v;
          bi = i;
        }
      };
      for (int c = c_first + tid; c < c_last; c += kRowThreads) {
        float v[EPC];
        F::unpack(*reinterpret_cast<const uint4 *>(row + (size_t)c * 16), v);
#pragma unroll
        for (int k = 0; k < EPC; ++k) best_of(v[k], c * EPC + k);
      }
      if (with_tail)
        for (int i = chunks * EPC + tid; i < vocab; i += kRowThreads) best_of(F::element(row, i), i);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (comes_first(ov, oi, bv, bi)) {
          bv = ov;
          bi = oi;
        }
      }
      if (lane == 0) {
        s_v[warp] = bv;
        s_i[warp] = bi;
      }
      __syncthreads();
      pv = s_v[0];
      pi = s_i[0];
#pragma unroll
      for (int q = 1; q < kRowThreads / 32; ++q)
        if (comes_first(s_v[q], s_i[q], pv, pi)) {
          pv = s_v[q];
          pi = s_i[q];
        }
      if (tid == 0 && pi != 0x7fffffff) mine[e] = top_key(pv, pi);
      __syncthreads();                               // s_v / s_i are free for the next round
    }
  }
  if (warp == 0) {                                   // the slice's (max, sum)
    m = lane < kRowThreads / 32 ? s_m[lane] : -INFINITY;
    s = lane < kRowThreads / 32 ? s_s[lane] : 0.f;
    const float own = m;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    s *= own == -INFINITY ? 0.f : __expf(own - m);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) mine[kMaxE] = (unsigned long long)__float_as_uint(m) << 32 | __float_as_uint(s);
  }
  __syncthreads();
  if (st.slices > 1) {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // every CTA is running, its barrier is set up
    if (st.rank > 0) {
      if (tid < E || tid == kMaxE) {
        const unsigned long long x = mine[tid];
        st_async_b32x2(map_to_cta(smem_u32(mine + tid), 0), (uint32_t)x, (uint32_t)(x >> 32), map_to_cta(st.bar, 0));
      }
      return;
    }
    bool landed = mbar_try_wait(st.bar, 0);
    if (!landed) {
      unsigned long long t0, t1;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
      do {                                           // at most 0.2 s
        landed = mbar_try_wait(st.bar, 0);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
      } while (!landed && t1 - t0 < 200000000ull);
    }
    if (!landed && tid == 0) flag_status(dev_status, b, TWIG_DEV_INTERNAL);
  }
  // ---- first CTA: the E best of the slices' lists, the row's log-sum-exp ----
  float M = -INFINITY, S = 0.f;
  if ((lane & 7) < st.slices) {
    const unsigned long long x = st.peer[(lane & 7) * kPeerStride + kMaxE];
    M = __uint_as_float((uint32_t)(x >> 32));
    S = __uint_as_float((uint32_t)x);
  }
  {
    const float own = M;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    S *= own == -INFINITY ? 0.f : __expf(own - M);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
  }
  const float lse = M + logf(S);
  if (tid < st.slices * E && (usable || u < 0)) {
    const int r = tid / E, e = tid - r * E;
    const unsigned long long x = st.peer[r * kPeerStride + e];
    int rank = e;                                    // (a list is in order)
    for (int q = 0; q < st.slices; ++q)
      if (q != r) {
        const ulonglong2 *list = reinterpret_cast<const ulonglong2 *>(st.peer + q * kPeerStride);
#pragma unroll
        for (int k = 0; k < kMaxE / 2; ++k) {
          const ulonglong2 y = list[k];
          rank += (y.x > x ? 1 : 0) + (y.y > x ? 1 : 0);
        }
      }
    if (x == 0) rank = E;                            // no entry
    if (rank < E) {
      const long long at = base + first + rank;      // (an unused slot's children: nobody selects them)
      node_tok[at] = usable ? top_index(x) : 0;
      node_parent[at] = usable ? u : -1;
      node_score[at] = usable ? parent_score + (top_value(x) - lse) : -INFINITY;
    }
  }
  __syncthreads();
}

// Grid (slices, rows, batch).  `ticket` (one counter per request, zero before the launch and zero again after
// it) selects the one-launch form: the request's last row to finish runs `tail`.
template <bool FP32>
__global__ void __launch_bounds__(kRowThreads)
tree_expand_kernel(const void *__restrict__ logits, long long row_stride, int vocab, int rows,
                   const int *__restrict__ src_node, int E, int level_base, int cap, int *node_tok,
                   int *node_parent, float *node_score, int *ticket, SelectArgs tail, int *dev_status) {
  extern __shared__ __align__(16) unsigned char work[];
  __shared__ __align__(16) unsigned long long s_peer[kMaxSlices * kPeerStride];
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ int s_last;
  const SliceTop st{s_peer, smem_u32(&s_bar), (int)blockIdx.x, (int)gridDim.x};
  const int r = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  // every list starts as "no entry" (a slice may hold fewer than E)
  for (int i = tid; i < kMaxSlices * kPeerStride; i += kRowThreads) s_peer[i] = 0;
  if (st.slices > 1) {
    __syncthreads();
    if (tid == 0) {
      mbar_init(st.bar, 1);
      mbar_arrive_expect_tx(st.bar, (uint32_t)(st.slices - 1) * (E + 1) * 8);
      mbar_init_fence_cluster();
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }
  grid_dependency_sync();
  const int u = src_node[(long long)b * rows + r];
  const int first = level_base + r * E;
  const long long base = (long long)b * cap;
  if (level_base == 1 && r == 0 && tid == 0 && st.rank == 0) {             // the first level also writes the root
    node_tok[base] = -1;
    node_parent[base] = -1;
    node_score[base] = 0.f;
  }
  const unsigned char *row = static_cast<const unsigned char *>(logits) + ((long long)b * rows + r) * row_stride * (FP32 ? 4 : 2);
  // (the host has checked that the level fits the state)
  expand_row<FP32>(row, vocab, E, st, u, level_base, base, first, node_tok, node_parent, node_score, dev_status, b);
  if (st.rank > 0) return;
  if (u >= level_base && tid == 0) flag_status(dev_status, b, TWIG_DEV_BAD_TREE);
  if (!ticket) return;
  // ---- the last row of the request to get here has every node of the level in view (a request with one
  // row has one cluster; expand_row ended with a CTA-wide barrier) ----
  if (rows > 1) {
    if (tid == 0) {
      int before;                                  // (the CTA's stores, ordered by the barrier, are released with it)
      asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(ticket + b) : "memory");
      s_last = before == rows - 1 ? 1 : 0;
      if (s_last) ticket[b] = 0;
    }
    __syncthreads();
    if (!s_last) return;
  }
  select_nodes(tail, b, cap, node_score, node_tok, node_parent, work, dev_status);
}

// Node 0 of every request: token -1, parent -1, score 0.
__global__ void tree_reset_kernel(int *node_tok, int *node_parent, float *node_score, int cap, int batch) {
  grid_dependency_sync();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  node_tok[(long long)b * cap] = -1;
  node_parent[(long long)b * cap] = -1;
  node_score[(long long)b * cap] = 0.f;
}

}  // namespace

}  // namespace twig

using namespace twig;


extern "C" twig_status tree_reset(int32_t *node_tok, int32_t *node_parent, float *node_score, int32_t cap,
                                  int32_t batch, void *stream) {
  if (!node_tok || !node_parent || !node_score) return TWIG_ERR_NULL;
  if (cap <= 0 || batch <= 0) return TWIG_ERR_SHAPE;
  PdlLaunch L(dim3((batch + 127) / 128), dim3(128), 0, static_cast<cudaStream_t>(stream));
  if (cudaLaunchKernelEx(&L.cfg, tree_reset_kernel, node_tok, node_parent, node_score, cap, batch) != cudaSuccess)
    return TWIG_ERR_CUDA;
  return launch_status();
}

namespace {

constexpr size_t kMaxSelectSmem = 48 * 1024;     // two words per node

twig_status check_expand(const void *logits, int logits_fp32, long long row_stride, int vocab, int rows,
                         const int *src_node, int n_children, int level_base, const int *node_tok,
                         const int *node_parent, const float *node_score, int cap, int batch) {
  if (!logits || !src_node || !node_tok || !node_parent || !node_score) return TWIG_ERR_NULL;
  if (vocab <= 0 || rows <= 0 || batch <= 0 || cap <= 0 || level_base <= 0 || row_stride < vocab) return TWIG_ERR_SHAPE;
  if (n_children <= 0 || n_children > kMaxE || n_children > vocab) return TWIG_ERR_UNSUPPORTED;
  if (batch > TWIG_MAX_BATCH || rows > 65535) return TWIG_ERR_UNSUPPORTED;
  if (level_base + (long long)rows * n_children > cap) return TWIG_ERR_SHAPE;
  const int esz = logits_fp32 ? 4 : 2;
  if (!aligned16(logits) || (row_stride * esz) % 16) return TWIG_ERR_ALIGN;
  return TWIG_OK;
}

// `ticket` == nullptr: the expansion alone.
twig_status launch_expand(const void *logits, int logits_fp32, long long row_stride, int vocab, int rows,
                          const int *src_node, int E, int level_base, int *node_tok, int *node_parent,
                          float *node_score, int cap, int batch, int *ticket, const SelectArgs &tail,
                          int *dev_status, cudaStream_t st) {
  const size_t smem = ticket ? (size_t)cap * 8 : 0;                  // the tail's two words per node
  static bool attr_set = false;                                      // (static arrays and a large state pass 48 KB)
  if (!attr_set) {
    if (cudaFuncSetAttribute(tree_expand_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSelectSmem) != cudaSuccess ||
        cudaFuncSetAttribute(tree_expand_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSelectSmem) != cudaSuccess)
      return TWIG_ERR_CUDA;
    attr_set = true;
  }
  // slices: at most a batch of loads per thread, so that the second pass need not read the slice again, and
  // further while four CTAs per SM hold all of them and a slice keeps two chunks per thread
  const int chunks = vocab / (logits_fp32 ? 4 : 8);
  int slices = 1;
  while (slices < kMaxSlices && (chunks > slices * kRowDeep * kRowThreads ||
                                 ((long long)rows * batch * slices * 2 <= 4 * 148 && chunks >= 4 * slices * kRowThreads)))
    slices *= 2;
  ClusterLaunch L(dim3(slices, rows, batch), dim3(kRowThreads), slices, st, smem);
  const cudaError_t err =
      logits_fp32 ? cudaLaunchKernelEx(&L.cfg, tree_expand_kernel<true>, logits, row_stride, vocab, rows, src_node, E,
                                       level_base, cap, node_tok, node_parent, node_score, ticket, tail, dev_status)
                  : cudaLaunchKernelEx(&L.cfg, tree_expand_kernel<false>, logits, row_stride, vocab, rows, src_node, E,
                                       level_base, cap, node_tok, node_parent, node_score, ticket, tail, dev_status);
  return err == cudaSuccess ? TWIG_OK : TWIG_ERR_CUDA;
}

twig_status launch_select(const float *node_score, const int32_t *node_tok, const int32_t *node_parent, int cap,
                          const SelectArgs &a, int batch, int *dev_status, cudaStream_t st) {
  const size_t smem = (size_t)cap * 8;
  if (smem > kMaxSelectSmem) return TWIG_ERR_UNSUPPORTED;
  PdlLaunch L(dim3(batch), dim3(kSelThreads), smem, st);
  if (cudaLaunchKernelEx(&L.cfg, tree_select_kernel, node_score, node_tok, node_parent, cap, a, dev_status) != cudaSuccess)
    return TWIG_ERR_CUDA;
  return launch_status();
}

twig_status expansion_args(int cap, int level_lo, int level_hi, int n_select, int *expand_node, int batch, SelectArgs *a) {
  if (!expand_node) return TWIG_ERR_NULL;
  if (cap <= 0 || batch <= 0 || n_select <= 0 || level_lo < 0 || level_hi <= level_lo || level_hi > cap)
    return TWIG_ERR_SHAPE;
  if (batch > TWIG_MAX_BATCH) return TWIG_ERR_UNSUPPORTED;
  if (n_select > level_hi - level_lo) return TWIG_ERR_SHAPE;     // every expansion row gets a node
  *a = SelectArgs{level_lo, level_hi, n_select, expand_node, n_select, nullptr, nullptr, nullptr, nullptr, 0};
  return TWIG_OK;
}

twig_status final_args(int cap, int n_built, int n_max, int *parent, int *draft_tok, int *n_nodes, int *kept_node,
                       int t_max, int batch, SelectArgs *a) {
  if (!parent || !draft_tok || !n_nodes) return TWIG_ERR_NULL;
  if (cap <= 0 || batch <= 0 || n_built <= 0 || n_built > cap || n_max <= 0 || t_max <= 0) return TWIG_ERR_SHAPE;
  if (n_max > t_max || t_max > TWIG_MAX_NODES || batch > TWIG_MAX_BATCH) return TWIG_ERR_UNSUPPORTED;
  *a = SelectArgs{1, n_built, n_max - 1, nullptr, 0, parent, draft_tok, n_nodes, kept_node, t_max};
  return TWIG_OK;
}

}  // namespace

extern "C" twig_status tree_expand_level(const void *logits, int32_t logits_fp32, int64_t row_stride,
                                         int32_t vocab, int32_t rows, const int32_t *src_node, int32_t n_children,
                                         int32_t level_base, int32_t *node_tok, int32_t *node_parent,
                                         float *node_score, int32_t cap, int32_t batch, int32_t *dev_status,
                                         void *stream) {
  const twig_status ok = check_expand(logits, logits_fp32, row_stride, vocab, rows, src_node, n_children, level_base,
                                      node_tok, node_parent, node_score, cap, batch);
  if (ok != TWIG_OK) return ok;
  return launch_expand(logits, logits_fp32, row_stride, vocab, rows, src_node, n_children, level_base, node_tok,
                       node_parent, node_score, cap, batch, nullptr, SelectArgs{}, dev_status,
                       static_cast<cudaStream_t>(stream));
}

extern "C" twig_status tree_select_expansion(const float *node_score, int32_t cap, int32_t level_lo, int32_t level_hi,
                                             int32_t n_select, int32_t *expand_node, int32_t batch,
                                             int32_t *dev_status, void *stream) {
  if (!node_score) return TWIG_ERR_NULL;
  SelectArgs a;
  const twig_status ok = expansion_args(cap, level_lo, level_hi, n_select, expand_node, batch, &a);
  if (ok != TWIG_OK) return ok;
  return launch_select(node_score, nullptr, nullptr, cap, a, batch, dev_status, static_cast<cudaStream_t>(stream));
}

extern "C" twig_status tree_finalize(const int32_t *node_tok, const int32_t *node_parent, const float *node_score,
                                     int32_t cap, int32_t n_built, int32_t n_max, int32_t *parent, int32_t *draft_tok,
                                     int32_t *n_nodes, int32_t *kept_node, int32_t t_max, int32_t batch,
                                     int32_t *dev_status, void *stream) {
  if (!node_tok || !node_parent || !node_score) return TWIG_ERR_NULL;
  SelectArgs a;
  const twig_status ok = final_args(cap, n_built, n_max, parent, draft_tok, n_nodes, kept_node, t_max, batch, &a);
  if (ok != TWIG_OK) return ok;
  return launch_select(node_score, node_tok, node_parent, cap, a, batch, dev_status, static_cast<cudaStream_t>(stream));
}

extern "C" twig_status tree_grow_level(const void *logits, int32_t logits_fp32, int64_t row_stride, int32_t vocab,
                                       int32_t rows, const int32_t *src_node, int32_t n_children, int32_t level_base,
                                       int32_t *node_tok, int32_t *node_parent, float *node_score, int32_t cap,
                                       int32_t batch, int32_t n_select, int32_t *expand_node, int32_t n_max,
                                       int32_t *parent, int32_t *draft_tok, int32_t *n_nodes, int32_t *kept_node,
                                       int32_t t_max, int32_t *ticket, int32_t *dev_status, void *stream) {
  twig_status ok = check_expand(logits, logits_fp32, row_stride, vocab, rows, src_node, n_children, level_base,
                                node_tok, node_parent, node_score, cap, batch);
  if (ok != TWIG_OK) return ok;
  if (!ticket) return TWIG_ERR_NULL;
  if ((size_t)cap * 8 > kMaxSelectSmem) return TWIG_ERR_UNSUPPORTED;
  const int level_hi = level_base + rows * n_children;
  SelectArgs a;
  ok = n_select > 0 ? expansion_args(cap, level_base, level_hi, n_select, expand_node, batch, &a)
                    : final_args(cap, level_hi, n_max, parent, draft_tok, n_nodes, kept_node, t_max, batch, &a);
  if (ok != TWIG_OK) return ok;
  return launch_expand(logits, logits_fp32, row_stride, vocab, rows, src_node, n_children, level_base, node_tok,
                       node_parent, node_score, cap, batch, ticket, a, dev_status, static_cast<cudaStream_t>(stream));
}
