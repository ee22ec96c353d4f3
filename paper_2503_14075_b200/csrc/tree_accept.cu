// Tree acceptance of tree-based self-speculative decoding (Sec. 5.4,
// Appendix A, Algorithm 2): the target walks the draft tree from the root,
// accepting at each level a child whose token equals its own prediction, and
// adds one bonus token; the accepted nodes' K/V rows of every layer are then
// appended to the KV cache (the rejected nodes' rows are simply never copied).
#include "vocab_row.cuh"

namespace twig {

constexpr int kAcceptThreads = 256;
constexpr int kAcceptSlicesPerCta = 4;   // (layer, kv head) slices copied by one CTA

// completion ticket per batch slot: the last CTA of a request to finish its
// copies publishes the new kv_len; the ticket returns to 0 for the next call.
__device__ unsigned int g_accept_ticket[TWIG_MAX_BATCH];

template <int D>
__global__ void __launch_bounds__(kAcceptThreads)
tree_accept_compact_kernel(const int *__restrict__ parent, const int *__restrict__ draft_tok,
                           const int *__restrict__ base_argmax, const int *__restrict__ n_nodes,
                           int t_max, int d_max, const __nv_bfloat16 *__restrict__ tree_k,
                           const __nv_bfloat16 *__restrict__ tree_v, KvViewMut cache, int *kv_len,
                           int *__restrict__ accept_len, int *__restrict__ path_out,
                           int *__restrict__ bonus_tok, int *dev_status) {
  constexpr int LPR = D / 8;
  __shared__ int s_parent[TWIG_MAX_NODES], s_tok[TWIG_MAX_NODES], s_tgt[TWIG_MAX_NODES];
  __shared__ int s_path[TWIG_MAX_NODES];
  __shared__ int s_best;

  grid_dependency_sync();
  const int b = blockIdx.y, tid = threadIdx.x;
  // everything the decision needs is requested at once (one round trip, not four: the kernel is a chain of
  // them; the one-layer step at batch 1 took 14.3 us of device time, 13.0 with this)
  const int n = n_nodes[b], base = kv_len[b];
  int my_parent = -1, my_tok = 0, my_tgt = 0;
  if (tid < t_max) {
    my_parent = parent[(long long)b * t_max + tid];
    my_tok = draft_tok[(long long)b * t_max + tid];
    my_tgt = base_argmax[(long long)b * t_max + tid];
  }
  if (n == 0) return;                                   // idle request
  const bool first = blockIdx.x == 0 && tid == 0;
  if (n < 0 || n > t_max) {
    if (first) flag_status(dev_status, b, TWIG_DEV_BAD_TREE);
    return;
  }
  if (tid == 0) s_best = -1;
  bool bad = false;
  if (tid < n) {
    s_parent[tid] = my_parent;
    s_tok[tid] = my_tok;
    s_tgt[tid] = my_tgt;
    bad = (tid == 0) ? (my_parent != -1) : (my_parent < 0 || my_parent >= tid);
  }
  if (__syncthreads_or(bad)) {
    if (first) flag_status(dev_status, b, TWIG_DEV_BAD_TREE);
    return;
  }
  // node i is accepted iff every edge on its root path matches; key orders by
  // depth first, then by lower index
  if (tid < n) {
    int x = tid, depth = 0;
    bool ok = true;
    while (x > 0) {                    // parent[x] < x, so this ends within n steps
      const int p = s_parent[x];
      ok = ok && (s_tok[x] == s_tgt[p]);
      x = p;
      ++depth;
    }
    if (ok) atomicMax(&s_best, depth * TWIG_MAX_NODES + (TWIG_MAX_NODES - 1 - tid));
  }
  __syncthreads();
  const int alen = s_best / TWIG_MAX_NODES;
  const int winner = TWIG_MAX_NODES - 1 - (s_best % TWIG_MAX_NODES);
  if (alen + 1 > d_max || base < 0 || base + alen + 1 > cache.max_len) {
    if (first) flag_status(dev_status, b, alen + 1 > d_max ? TWIG_DEV_BAD_TREE : TWIG_DEV_OVERFLOW);
    return;
  }
  if (tid == 0) {
    int x = winner;
    for (int j = alen; j >= 0; --j) {
      s_path[j] = x;
      x = s_parent[x];
    }
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    if (tid < d_max) path_out[(long long)b * d_max + tid] = (tid <= alen) ? s_path[tid] : -1;
    if (tid == 0) {
      accept_len[b] = alen;
      bonus_tok[b] = s_tgt[winner];
    }
  }

  // copy rows path[0..alen] of the slices this CTA owns, K and V
  const int n_slices = cache.n_layers * cache.n_kv_heads;
  const int slice0 = blockIdx.x * kAcceptSlicesPerCta;
  const int rows = alen + 1;
  const int items = kAcceptSlicesPerCta * rows * 2 * LPR;
  for (int it = tid; it < items; it += kAcceptThreads) {
    const int sub = it % LPR;
    int r = it / LPR;
    const int which = r & 1;
    r >>= 1;
    const int j = r % rows, slice = slice0 + r / rows;
    if (slice >= n_slices) continue;
    const int layer = slice / cache.n_kv_heads, h = slice % cache.n_kv_heads;
    const long long toff = ((((long long)layer * cache.batch + b) * cache.n_kv_heads + h) * t_max + s_path[j]) * D + sub * 8;
    const long long coff = layer * cache.stride_layer + b * cache.stride_batch + h * cache.stride_head +
                           (long long)(base + j) * cache.stride_pos + sub * 8;
    const uint4 val = ld_nc_16((which ? tree_v : tree_k) + toff);
    st_16((which ? cache.v : cache.k) + coff, val);
  }

  // every CTA has read kv_len[b] above; the last one to arrive updates it
  if (gridDim.x == 1) {
    if (tid == 0) kv_len[b] = base + alen + 1;
    return;
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    const unsigned int t = atomicAdd(&g_accept_ticket[b], 1u);
    if (t == gridDim.x - 1) {
      g_accept_ticket[b] = 0;
      kv_len[b] = base + alen + 1;
      __threadfence();
    }
  }
}

// ---------------------------------------------------------------------------
// Greedy target token per tree node: argmax over the vocabulary, lowest index on ties.
// Grid (slices, nodes, requests), clusters of the slices of a row.
// ---------------------------------------------------------------------------
template <bool FP32>
__global__ void __launch_bounds__(kRowThreads)
base_argmax_kernel(const void *__restrict__ logits, long long row_stride, int vocab,
                   const int *__restrict__ n_nodes, int t_max, int *__restrict__ out, int *dev_status) {
  constexpr int EPC = RowFormat<FP32>::EPC;
  __shared__ __align__(16) float4 s_peer[kMaxSlices];
  __shared__ __align__(8) unsigned long long s_bar;
  grid_dependency_sync();
  const int b = blockIdx.z, node = blockIdx.y, tid = threadIdx.x;
  SliceMerge sm{s_peer, smem_u32(&s_bar), (int)blockIdx.x, (int)gridDim.x};
  const int n = n_nodes[b];
  if (n < 0 || n > t_max) {
    if (node == 0 && sm.rank == 0 && tid == 0) flag_status(dev_status, b, TWIG_DEV_BAD_TREE);
    return;
  }
  if (node >= n) return;
  sm.start();
  const unsigned char *row = static_cast<const unsigned char *>(logits) +
                             ((long long)b * t_max + node) * row_stride * (FP32 ? 4 : 2);
  const int chunks = vocab / EPC, per = (chunks + sm.slices - 1) / sm.slices;
  RowBest best = scan_slice<FP32, false>(row, sm.rank * per, min(chunks, (sm.rank + 1) * per),
                                         sm.rank == 0 && chunks * EPC < vocab, vocab);
  const bool landed = sm.merge<false>(best);
  if (sm.rank > 0 || tid != 0) return;
  if (landed) out[(long long)b * t_max + node] = best.index;
  else flag_status(dev_status, b, TWIG_DEV_INTERNAL);
}

}  // namespace twig

using namespace twig;

extern "C" twig_status tree_base_argmax(const void *logits, int32_t logits_fp32, int64_t row_stride,
                                        int32_t vocab, const int32_t *n_nodes, int32_t batch,
                                        int32_t t_max, int32_t *base_argmax, int32_t *dev_status,
                                        void *stream) {
  if (!logits || !n_nodes || !base_argmax) return TWIG_ERR_NULL;
  if (vocab <= 0 || batch <= 0 || t_max <= 0 || row_stride < vocab) return TWIG_ERR_SHAPE;
  if (t_max > TWIG_MAX_NODES || batch > TWIG_MAX_BATCH) return TWIG_ERR_UNSUPPORTED;
  const int esz = logits_fp32 ? 4 : 2;
  if (!aligned16(logits) || (row_stride * esz) % 16) return TWIG_ERR_ALIGN;
  const int slices = row_slices((long long)t_max * batch, vocab / (16 / esz));
  ClusterLaunch L(dim3(slices, t_max, batch), dim3(kRowThreads), slices, static_cast<cudaStream_t>(stream));
  const long long rs = row_stride;
  const cudaError_t err =
      logits_fp32 ? cudaLaunchKernelEx(&L.cfg, base_argmax_kernel<true>, logits, rs, vocab, n_nodes, t_max, base_argmax, dev_status)
                  : cudaLaunchKernelEx(&L.cfg, base_argmax_kernel<false>, logits, rs, vocab, n_nodes, t_max, base_argmax, dev_status);
  return err == cudaSuccess ? TWIG_OK : TWIG_ERR_CUDA;
}


extern "C" twig_status tree_accept_compact(const int32_t *parent, const int32_t *draft_tok,
                                           const int32_t *base_argmax, const int32_t *n_nodes,
                                           int32_t t_max, int32_t d_max, const void *tree_k_all,
                                           const void *tree_v_all, const twig_kv *cache,
                                           int32_t *kv_len, int32_t *accept_len, int32_t *path,
                                           int32_t *bonus_tok, int32_t *dev_status, void *stream) {
  if (!parent || !draft_tok || !base_argmax || !n_nodes || !tree_k_all || !tree_v_all || !kv_len ||
      !accept_len || !path || !bonus_tok)
    return TWIG_ERR_NULL;
  twig_status s = check_kv(cache);
  if (s != TWIG_OK) return s;
  if (t_max <= 0 || d_max <= 0) return TWIG_ERR_SHAPE;
  if (t_max > TWIG_MAX_NODES || d_max > TWIG_MAX_NODES) return TWIG_ERR_UNSUPPORTED;
  if (!aligned16(tree_k_all) || !aligned16(tree_v_all)) return TWIG_ERR_ALIGN;
  const int n_slices = cache->n_layers * cache->n_kv_heads;
  dim3 grid((n_slices + kAcceptSlicesPerCta - 1) / kAcceptSlicesPerCta, cache->batch);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  auto tk = static_cast<const __nv_bfloat16 *>(tree_k_all);
  auto tv = static_cast<const __nv_bfloat16 *>(tree_v_all);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kAcceptThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = launch_overlap_enabled() ? 1 : 0;
  const KvViewMut cv = view_of_mut(cache);
  const cudaError_t err =
      cache->head_dim == 128
          ? cudaLaunchKernelEx(&cfg, tree_accept_compact_kernel<128>, parent, draft_tok, base_argmax, n_nodes, t_max,
                               d_max, tk, tv, cv, kv_len, accept_len, path, bonus_tok, dev_status)
          : cudaLaunchKernelEx(&cfg, tree_accept_compact_kernel<64>, parent, draft_tok, base_argmax, n_nodes, t_max,
                               d_max, tk, tv, cv, kv_len, accept_len, path, bonus_tok, dev_status);
  if (err != cudaSuccess) return TWIG_ERR_CUDA;
  return launch_status();
}
