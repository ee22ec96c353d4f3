// Chain drafting of sequence self-speculative decoding with its early exit (Appendix A,
// "Self-speculative decoding"; Algorithm 1's draft loop): the draft model predicts up to
// delta tokens one after another and stops early once the probability of the token it has
// just predicted falls below theta; that token still belongs to the draft.  The draft model
// runs between the calls (its logits are inputs); one call takes one draft distribution per
// request, picks the greedy token (lowest id among equal logits), computes its probability,
// appends it to the request's chain (node n's parent is node n - 1, the layout tree attention
// and acceptance take: a chain is a tree) and decides whether the request goes on drafting.
// Requests that have stopped ignore further calls, so a batch can be driven through delta
// calls without reading anything back.
#include "vocab_row.cuh"

namespace twig {

// Grid (slices, batch), clusters of the slices of a row.  One CTA per row took 13 us from a cold start at
// 32000 fp32 logits (four round trips of loads, then one exponential after the other).
template <bool FP32>
__global__ void __launch_bounds__(kRowThreads)
chain_draft_step_kernel(const void *__restrict__ logits, long long row_stride, int vocab, int max_draft,
                        float threshold, int *parent, int *draft_tok, float *tok_prob, int *n_nodes, int *active,
                        int t_max, int *dev_status) {
  constexpr int EPC = RowFormat<FP32>::EPC;
  __shared__ __align__(16) float4 s_peer[kMaxSlices];
  __shared__ __align__(8) unsigned long long s_bar;
  grid_dependency_sync();
  const int b = blockIdx.y, tid = threadIdx.x;
  SliceMerge sm{s_peer, smem_u32(&s_bar), (int)blockIdx.x, (int)gridDim.x};
  const bool go = active[b] != 0;
  const int n = n_nodes[b];
  if (!go) return;
  const bool room = n >= 1 && n < t_max;            // a root, and room for another node
  RowBest best{-INFINITY, 0.f, 0};
  bool landed = true;
  // (both words were read before the first CTA below can write them: it waits for its peers' results)
  if (room) {
    sm.start();
    const unsigned char *row = static_cast<const unsigned char *>(logits) + (long long)b * row_stride * (FP32 ? 4 : 2);
    const int chunks = vocab / EPC, per = (chunks + sm.slices - 1) / sm.slices;
    best = scan_slice<FP32, true>(row, sm.rank * per, min(chunks, (sm.rank + 1) * per),
                                  sm.rank == 0 && chunks * EPC < vocab, vocab);
    landed = sm.merge<true>(best);
  }
  if (sm.rank > 0 || tid != 0) return;
  if (!room || !landed) {
    flag_status(dev_status, b, room ? TWIG_DEV_INTERNAL : TWIG_DEV_BAD_TREE);
    active[b] = 0;
    return;
  }
  const float prob = 1.f / best.s;                  // softmax(row)[token]: the token's logit is the maximum
  const long long at = (long long)b * t_max + n;
  parent[at] = n - 1;
  draft_tok[at] = best.index;
  if (tok_prob) tok_prob[at] = prob;
  n_nodes[b] = n + 1;
  // n draft tokens now (the root is node 0): stop at delta of them or below the confidence threshold
  if (n >= max_draft || prob < threshold) active[b] = 0;
}

__global__ void chain_draft_reset_kernel(int *parent, int *draft_tok, float *tok_prob, int *n_nodes, int *active,
                                         int t_max, int batch) {
  grid_dependency_sync();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < batch * t_max) {
    parent[idx] = -1;
    draft_tok[idx] = idx % t_max == 0 ? -1 : 0;
    if (tok_prob) tok_prob[idx] = idx % t_max == 0 ? 1.f : 0.f;
  }
  if (idx < batch) {
    n_nodes[idx] = 1;        // the root: the last accepted token
    active[idx] = 1;
  }
}

}  // namespace twig

using namespace twig;

extern "C" twig_status chain_draft_reset(int32_t *parent, int32_t *draft_tok, float *tok_prob, int32_t *n_nodes,
                                         int32_t *active, int32_t t_max, int32_t batch, void *stream) {
  if (!parent || !draft_tok || !n_nodes || !active) return TWIG_ERR_NULL;
  if (t_max <= 0 || batch <= 0) return TWIG_ERR_SHAPE;
  if (t_max > TWIG_MAX_NODES || batch > TWIG_MAX_BATCH) return TWIG_ERR_UNSUPPORTED;
  const int total = batch * t_max;
  PdlLaunch L(dim3((total + 255) / 256), dim3(256), 0, static_cast<cudaStream_t>(stream));
  return cudaLaunchKernelEx(&L.cfg, chain_draft_reset_kernel, parent, draft_tok, tok_prob, n_nodes, active, t_max, batch) ==
                 cudaSuccess
             ? TWIG_OK
             : TWIG_ERR_CUDA;
}

extern "C" twig_status chain_draft_step(const void *logits, int32_t logits_fp32, int64_t row_stride, int32_t vocab,
                                        int32_t max_draft, float threshold, int32_t *parent, int32_t *draft_tok,
                                        float *tok_prob, int32_t *n_nodes, int32_t *active, int32_t t_max,
                                        int32_t batch, int32_t *dev_status, void *stream) {
  if (!logits || !parent || !draft_tok || !n_nodes || !active) return TWIG_ERR_NULL;
  if (vocab <= 0 || batch <= 0 || t_max <= 0 || row_stride < vocab || max_draft <= 0) return TWIG_ERR_SHAPE;
  if (max_draft + 1 > t_max) return TWIG_ERR_SHAPE;            // the root and delta draft tokens must fit
  if (t_max > TWIG_MAX_NODES || batch > TWIG_MAX_BATCH) return TWIG_ERR_UNSUPPORTED;
  if (!(threshold >= 0.f)) return TWIG_ERR_SHAPE;               // (also refuses NaN)
  const int esz = logits_fp32 ? 4 : 2;
  if (!aligned16(logits) || (row_stride * esz) % 16) return TWIG_ERR_ALIGN;
  const int slices = row_slices(batch, vocab / (16 / esz));
  ClusterLaunch L(dim3(slices, batch), dim3(kRowThreads), slices, static_cast<cudaStream_t>(stream));
  const long long rs = row_stride;
  const cudaError_t err =
      logits_fp32 ? cudaLaunchKernelEx(&L.cfg, chain_draft_step_kernel<true>, logits, rs, vocab, max_draft, threshold, parent,
                                       draft_tok, tok_prob, n_nodes, active, t_max, dev_status)
                  : cudaLaunchKernelEx(&L.cfg, chain_draft_step_kernel<false>, logits, rs, vocab, max_draft, threshold, parent,
                                       draft_tok, tok_prob, n_nodes, active, t_max, dev_status);
  return err == cudaSuccess ? TWIG_OK : TWIG_ERR_CUDA;
}
