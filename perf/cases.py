"""The work that users have this library do, as cases that can be timed and compared.

Five kinds, each a part of serving a vision-language model with a twig:

  prune   after prefill: score the visual tokens, keep the best, compact the KV cache of all layers
  guide   the other two scoring guides: P-Head scores that prune layer-K hidden states, and the
          multi-query text-to-visual guide
  tree    drafting, tree form: grow a token tree level by level and cut it to verification layout
  chain   drafting, sequence form: greedy draft tokens with the early exit
  verify  one verification step: tree attention in every layer, the target's greedy tokens,
          acceptance and the KV append

The shapes are those of the benchmark's configurations and of the tests; `draw` covers the ranges
between and around them.  Tokens, trees and lengths are drawn like those of `synth`, tensors are
made on the GPU.
"""
import math
import random

import numpy as np
import torch

from paper_2503_14075_b200 import synth
from paper_2503_14075_b200 import twig as tw

DEV = "cuda"


def listed():
    return [
        # one layer of the smallest configuration: latency of a handful of calls, head_dim 64
        dict(name="verify-tiny", kind="verify", batch=1, layers=1, q_heads=4, kv_heads=4, head_dim=64, nodes=8,
             kv_len=64, ragged=False, vocab=32000, fp32=False),
        # a single user's decoding step (7B, pruned prompt and some answer in the cache)
        dict(name="verify-b1", kind="verify", batch=1, layers=32, q_heads=32, kv_heads=32, head_dim=128, nodes=26,
             kv_len=227, ragged=False, vocab=32000, fp32=True),
        # continuous batching: sixteen requests of different lengths, trees of different sizes
        dict(name="verify-b16-ragged", kind="verify", batch=16, layers=32, q_heads=32, kv_heads=32, head_dim=128,
             nodes=32, kv_len=463, ragged=True, vocab=32000, fp32=False),
        # high-resolution images, long answers, full trees
        dict(name="verify-hires-b4", kind="verify", batch=4, layers=32, q_heads=32, kv_heads=32, head_dim=128,
             nodes=64, kv_len=1472, ragged=False, vocab=32000, fp32=False),
        # grouped-query model with a long cache: the largest step
        dict(name="verify-gqa-b8-8k", kind="verify", batch=8, layers=28, q_heads=28, kv_heads=4, head_dim=128,
             nodes=64, kv_len=8128, ragged=False, vocab=32000, fp32=False),
        # time to first token of one request
        dict(name="prune-b1", kind="prune", batch=1, layers=32, q_heads=32, kv_heads=32, head_dim=128, text=99,
             visual=576, keep=64, in_place=False, scope=0, ragged=False),
        # a prefill batch compacted where it lies (no second cache)
        dict(name="prune-b16-inplace", kind="prune", batch=16, layers=32, q_heads=32, kv_heads=32, head_dim=128,
             text=200, visual=576, keep=192, in_place=True, scope=0, ragged=True),
        # high-resolution prompts, most of the image dropped
        dict(name="prune-hires-b4", kind="prune", batch=4, layers=32, q_heads=32, kv_heads=32, head_dim=128, text=128,
             visual=2880, keep=320, in_place=False, scope=1, ragged=False),
        # P-Head scores with both gates, then the hidden states of layer K
        dict(name="phead-hires-b4", kind="guide", guide="gated", batch=4, q_heads=32, kv_heads=32, head_dim=128,
             text=128, visual=2880, keep=320, width=4096, ragged=False),
        # the guide summed over the text tokens after the image
        dict(name="text-guide-hires-b4", kind="guide", guide="text", batch=4, q_heads=32, kv_heads=32, head_dim=128,
             text=128, visual=2880, keep=320, width=4096, ragged=False),
        # token trees of a batch, the paper's E = K = 10, D = 4, N_max = 60
        dict(name="tree-b16", kind="tree", batch=16, vocab=32000, width=10, select=10, depth=4, n_max=60, fp32=False),
        # a single user's chain draft, delta = 5, theta = 0.6
        dict(name="chain-b1", kind="chain", batch=1, vocab=32000, delta=5, fp32=True),
    ]


# ---- draws -----------------------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(["verify", "verify", "verify", "prune", "prune", "guide", "tree", "chain"])
    q_heads, kv_heads, head_dim = rng.choice([(32, 32, 128), (32, 32, 128), (28, 4, 128), (32, 8, 128), (16, 16, 64), (4, 4, 64)])
    heads = dict(q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim)
    if kind == "verify":
        return dict(kind=kind, batch=_log_int(rng, 1, 16), layers=_log_int(rng, 1, 32), **heads,
                    nodes=_log_int(rng, 4, 64), kv_len=_log_int(rng, 32, 8128), ragged=rng.random() < 0.5,
                    vocab=_log_int(rng, 8000, 130000), fp32=rng.random() < 0.5)
    visual = _log_int(rng, 100, 4096)
    image = dict(text=_log_int(rng, 20, 500), visual=visual, keep=max(1, int(visual * rng.uniform(0.04, 0.5))),
                 ragged=rng.random() < 0.5)
    if kind == "prune":
        return dict(kind=kind, batch=_log_int(rng, 1, 16), layers=_log_int(rng, 1, 32), **heads, **image,
                    in_place=rng.random() < 0.4, scope=rng.randint(0, 1))
    if kind == "guide":
        return dict(kind=kind, guide=rng.choice(["gated", "text"]), batch=_log_int(rng, 1, 8), **heads, **image,
                    width=8 * _log_int(rng, 128, 1024))
    if kind == "tree":
        width = rng.randint(2, 16)
        return dict(kind=kind, batch=_log_int(rng, 1, 32), vocab=_log_int(rng, 8000, 130000), width=width,
                    select=rng.randint(1, width), depth=rng.randint(2, 6), n_max=rng.randint(8, 64),
                    fp32=rng.random() < 0.5)
    return dict(kind=kind, batch=_log_int(rng, 1, 64), vocab=_log_int(rng, 8000, 130000), delta=rng.randint(2, 8),
                fp32=rng.random() < 0.5)


def _footprint(case):
    """Bytes of a case's own KV caches."""
    if case["kind"] == "verify":
        rows = case["kv_len"] + case["nodes"]
    elif case["kind"] == "prune":
        rows = case["text"] + case["visual"] + (0 if case["in_place"] else case["text"] + case["keep"])
    else:
        return 0
    return 4 * case["layers"] * case["batch"] * case["kv_heads"] * case["head_dim"] * rows


def draw(rng):
    while True:
        case = _draw_once(rng)
        w = work(case)
        if w["bytes"] <= 2.5e9 and w["flops"] <= 8e11 and _footprint(case) <= 7e9:
            return case


# ---- what a case's requests look like ---------------------------------------------------------------
def _requests(case):
    """Per-request (lengths ...) of a case: the case's own figures are the largest request's.  They are
    part of the case, the same for every seed."""
    rng = random.Random(sum(case[k] * p for k, p in (("batch", 7919), ("q_heads", 104729))))
    spread = (lambda hi, lo: rng.randint(lo, hi)) if case["ragged"] else (lambda hi, lo: hi)
    reqs = []
    for b in range(case["batch"]):
        if case["kind"] == "verify":
            reqs.append((case["kv_len"], case["nodes"]) if b == 0 else
                        (spread(case["kv_len"], (case["kv_len"] + 1) // 2), spread(case["nodes"], (case["nodes"] + 1) // 2)))
        else:
            text = case["text"] if b == 0 else spread(case["text"], max(2, case["text"] // 4))
            keep = case["keep"] if b == 0 else spread(case["keep"], max(1, case["keep"] // 3))
            before = min(64, text // 2)
            reqs.append((before, case["visual"], text - before, keep))
    return reqs


def _i32(x):
    return torch.tensor(np.ascontiguousarray(x, dtype=np.int32), device=DEV)


class _Maker:
    def __init__(self, seed):
        self.gen = torch.Generator(device=DEV)
        self.gen.manual_seed(seed)

    def normal(self, shape, std=1.0, dtype=torch.bfloat16):
        x = torch.empty(shape, dtype=dtype, device=DEV)
        return x.normal_(0.0, std, generator=self.gen)

    def uniform(self, shape, lo, hi):
        return torch.empty(shape, dtype=torch.float32, device=DEV).uniform_(lo, hi, generator=self.gen)

    def logits(self, shape, fp32, lead):
        """Logits as a language-model head gives them: a broad bulk and `lead` likely tokens per row; rows
        padded to 16 bytes.  Returns (logits, the likely tokens)."""
        *outer, vocab = shape
        full = self.normal((*outer, (vocab + 7) // 8 * 8), 1.5, torch.float32 if fp32 else torch.bfloat16)
        x = full[..., :vocab]
        top = torch.randint(0, vocab, (*outer, lead), generator=self.gen, device=DEV)
        x.scatter_(-1, top, self.uniform((*outer, lead), 9.0, 16.0).to(x.dtype))
        return x, top


# ---- prepare ------------------------------------------------------------------------------------------
def _prepare_verify(case, m, rng):
    B, nl, Hq, Hkv, d, T = (case[k] for k in ("batch", "layers", "q_heads", "kv_heads", "head_dim", "nodes"))
    V, reqs = case["vocab"], _requests(case)
    kv_len, n_nodes = [r[0] for r in reqs], [r[1] for r in reqs]
    parent = np.full((B, T), -1, dtype=np.int32)
    draft = np.zeros((B, T), dtype=np.int32)
    target = np.zeros((B, T), dtype=np.int64)
    for b, n in enumerate(n_nodes):
        par = synth.random_tree(rng, n, int(rng.integers(3, 7)))
        parent[b, :n] = par
        target[b] = rng.integers(0, V, T)
        # siblings carry distinct tokens; with probability 0.65 one of them is the target's
        draft[b, :n] = (target[b, par] + 1 + np.arange(n)) % V
        for u in range(n):
            kids = np.nonzero(par == u)[0]
            if len(kids) and rng.random() < 0.65:
                draft[b, kids[rng.integers(len(kids))]] = target[b, u]
    logits, _ = m.logits((B, T, V), case["fp32"], 4)
    logits.scatter_(-1, torch.from_numpy(target)[..., None].to(DEV), 20.0)
    max_len = (case["kv_len"] + T + 31) // 32 * 32
    k, v = m.normal((nl, B, Hkv, max_len, d)), m.normal((nl, B, Hkv, max_len, d))
    q, tree_k, tree_v = m.normal((nl, B, T, Hq, d)), m.normal((nl, B, Hkv, T, d)), m.normal((nl, B, Hkv, T, d))
    out = torch.zeros_like(q)
    zeros = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)  # noqa: E731
    return dict(case=case, q=list(q), tree_k=list(tree_k), tree_v=list(tree_v), out=list(out), out_all=out,
                tree_k_all=tree_k, tree_v_all=tree_v, cache=tw.KV.of(k, v), k=k, v=v, start_len=_i32(kv_len),
                kv_len=_i32(kv_len), n_nodes=_i32(n_nodes), parent=_i32(parent), draft=_i32(draft), logits=logits,
                target=zeros(B, T), accept_len=zeros(B), path=zeros(B, T), bonus=zeros(B), status=zeros(B))


def _prompt(case, m):
    """The prompts' layout, and the scoring queries and keys: some image tokens draw much of the attention,
    most of them little."""
    B, Hq, Hkv, d = (case[k] for k in ("batch", "q_heads", "kv_heads", "head_dim"))
    reqs = _requests(case)
    length = max(a + n + c for a, n, c, _ in reqs)
    s = dict(case=case, prefix_len=_i32([a + n + c for a, n, c, _ in reqs]), vis_start=_i32([r[0] for r in reqs]),
             n_vis=_i32([r[1] for r in reqs]), keep=_i32([r[3] for r in reqs]), length=length,
             scores=torch.zeros((B, case["visual"]), dtype=torch.float32, device=DEV),
             kept=torch.full((B, case["keep"]), -1, dtype=torch.int32, device=DEV),
             new_len=torch.zeros(B, dtype=torch.int32, device=DEV), status=torch.zeros(B, dtype=torch.int32, device=DEV))
    q = m.normal((B, Hq, d))
    k = m.normal((B, Hkv, length, d))
    salience = m.normal((B, 1, length, 1), 1.5, torch.float32)
    k += (salience * q.float().view(B, Hkv, Hq // Hkv, d).sum(2)[:, :, None, :] / d ** 0.5).to(torch.bfloat16)
    s.update(twig_q=q, twig_k=k)
    return s


def _prepare_prune(case, m, rng):
    s = _prompt(case, m)
    B, nl, Hkv, d = (case[k] for k in ("batch", "layers", "kv_heads", "head_dim"))
    shape = (nl, B, Hkv, s["length"], d)
    k, v = m.normal(shape), m.normal(shape)
    s["src"] = tw.KV.of(k, v)
    s["pos"] = torch.arange(s["length"], dtype=torch.int32, device=DEV).repeat(B, 1)
    if case["in_place"]:
        s.update(dst=s["src"], k=k, v=v, pos_out=s["pos"])
    else:
        room = (case["text"] + case["keep"] + 31) // 32 * 32
        dk = torch.zeros((nl, B, Hkv, room, d), dtype=torch.bfloat16, device=DEV)
        dv = torch.zeros_like(dk)
        s.update(dst=tw.KV.of(dk, dv), k=dk, v=dv, pos_out=torch.zeros_like(s["pos"]))
    s["ws"] = torch.empty(tw.twig_workspace_bytes(B, case["q_heads"], d, s["length"], 64), dtype=torch.uint8, device=DEV)
    return s


def _prepare_guide(case, m, rng):
    s = _prompt(case, m)
    B, Hq, d = (case[k] for k in ("batch", "q_heads", "head_dim"))
    if case["guide"] == "gated":
        s["q_gate"] = torch.sigmoid(m.normal(s["twig_q"].shape)).mul_(2)
        s["k_gate"] = torch.sigmoid(m.normal(s["twig_k"].shape)).mul_(2)
        s["hidden"] = m.normal((B, s["length"], case["width"]))
        s["pruned"] = torch.zeros((B, case["text"] + case["keep"], case["width"]), dtype=torch.bfloat16, device=DEV)
        s["ws"] = torch.empty(tw.twig_workspace_bytes(B, Hq, d, s["length"], 64), dtype=torch.uint8, device=DEV)
    else:
        # one query row per text token after the image, all of them near the question's direction
        n_text = max(c for _, _, c, _ in _requests(case))
        s["q_text"] = (0.7 * s["twig_q"][:, :, None, :] + m.normal((B, Hq, n_text, d), 0.7)).contiguous()
        need = tw.ttp_multiquery_workspace_bytes(B, Hq, n_text, case["visual"], s["length"])
        s["ws"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    return s


def _prepare_tree(case, m, rng):
    B, E, K, D = (case[k] for k in ("batch", "width", "select", "depth"))
    levels = [1] + [K] * (D - 1)          # draft rows per level
    zeros = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)  # noqa: E731
    return dict(case=case, logits=[m.logits((B, rows, case["vocab"]), case["fp32"], 24)[0] for rows in levels],
                state=tw.TreeState(B, 1 + E * sum(levels), DEV), root=zeros(B, 1), expand=[zeros(B, K) for _ in levels[1:]],
                parent=zeros(B, case["n_max"]), draft=zeros(B, case["n_max"]), n_nodes=zeros(B), status=zeros(B))


def _prepare_chain(case, m, rng):
    B, t_max = case["batch"], case["delta"] + 1
    zeros = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)  # noqa: E731
    return dict(case=case, logits=[m.logits((B, case["vocab"]), case["fp32"], 3)[0] for _ in range(case["delta"])],
                parent=zeros(B, t_max), draft=zeros(B, t_max), n_nodes=zeros(B), active=zeros(B), status=zeros(B),
                prob=torch.zeros((B, t_max), dtype=torch.float32, device=DEV))


def prepare(case, seed):
    make = dict(verify=_prepare_verify, prune=_prepare_prune, guide=_prepare_guide, tree=_prepare_tree, chain=_prepare_chain)
    return make[case["kind"]](case, _Maker(seed), np.random.default_rng(seed))


# ---- run ----------------------------------------------------------------------------------------------
# the layers after the first follow another layer's attention, which leaves lengths and cache alone
_FIRST, _LATER = tw.attn_flags(), tw.attn_flags(early_prefix=True)


def _run_verify(s):
    s["kv_len"].copy_(s["start_len"])     # the step's lengths (acceptance moves them on)
    cache, kv_len, n_nodes, parent, status = s["cache"], s["kv_len"], s["n_nodes"], s["parent"], s["status"]
    for layer, (q, tk, tv, out) in enumerate(zip(s["q"], s["tree_k"], s["tree_v"], s["out"])):
        tw.tree_verify_attention(q, tk, tv, cache, layer, kv_len, n_nodes, parent, out, dev_status=status,
                                 flags=_LATER if layer else _FIRST)
    tw.tree_base_argmax(s["logits"], n_nodes, s["target"], dev_status=status)
    tw.tree_accept_compact(parent, s["draft"], s["target"], n_nodes, s["tree_k_all"], s["tree_v_all"], cache, kv_len,
                           s["accept_len"], s["path"], s["bonus"], dev_status=status)
    return {key: s[key] for key in ("out_all", "target", "accept_len", "path", "bonus", "kv_len", "k", "v", "status")}


def _run_prune(s):
    tw.ttp_score_topk_compact(s["twig_q"], s["twig_k"], s["prefix_len"], s["vis_start"], s["n_vis"], s["keep"],
                              s["scores"], s["kept"], s["src"], s["dst"], s["ws"], pos_in=s["pos"], pos_out=s["pos_out"],
                              new_len=s["new_len"], norm_scope=s["case"]["scope"], dev_status=s["status"])
    return {key: s[key] for key in ("scores", "kept", "k", "v", "pos_out", "new_len", "status")}


def _run_guide(s):
    layout = (s["prefix_len"], s["vis_start"], s["n_vis"])
    if s["case"]["guide"] == "text":
        tw.ttp_score_multiquery(s["q_text"], s["twig_k"], *layout, s["scores"], s["ws"], dev_status=s["status"])
        return {key: s[key] for key in ("scores", "status")}
    tw.ttp_score_gated(s["twig_q"], s["q_gate"], s["twig_k"], s["k_gate"], *layout, s["scores"], s["ws"],
                       dev_status=s["status"])
    tw.ttp_topk(s["scores"], s["n_vis"], s["keep"], s["kept"], dev_status=s["status"])
    tw.ttp_compact_rows(s["hidden"], s["pruned"], s["kept"], s["keep"], *layout, new_len=s["new_len"],
                        dev_status=s["status"])
    return {key: s[key] for key in ("scores", "kept", "pruned", "new_len", "status")}


def _run_tree(s):
    case, state = s["case"], s["state"]
    E, n_levels = case["width"], case["depth"]
    base, src = 1, s["root"]
    for level, logits in enumerate(s["logits"]):
        if level < n_levels - 1:
            tw.tree_grow_level(logits, src, E, base, state, expand_node=s["expand"][level], dev_status=s["status"])
            base, src = base + logits.shape[1] * E, s["expand"][level]
        else:
            tw.tree_grow_level(logits, src, E, base, state, n_max=case["n_max"], parent=s["parent"],
                               draft_tok=s["draft"], n_nodes=s["n_nodes"], dev_status=s["status"])
    return dict(tok=state.tok, par=state.parent, score=state.score, expand=s["expand"], parent=s["parent"],
                draft=s["draft"], n_nodes=s["n_nodes"], status=s["status"])


def _run_chain(s):
    chain = (s["parent"], s["draft"], s["n_nodes"], s["active"])
    tw.chain_draft_reset(*chain, tok_prob=s["prob"])
    for logits in s["logits"]:
        tw.chain_draft_step(logits, s["case"]["delta"], 0.6, *chain, tok_prob=s["prob"], dev_status=s["status"])
    return {key: s[key] for key in ("parent", "draft", "n_nodes", "active", "prob", "status")}


_RUN = dict(verify=_run_verify, prune=_run_prune, guide=_run_guide, tree=_run_tree, chain=_run_chain)


def run(state):
    return _RUN[state["case"]["kind"]](state)


# ---- what a pass cannot do without ----------------------------------------------------------------------
def work(case):
    B, kind = case["batch"], case["kind"]
    if kind in ("tree", "chain"):
        rows = case["delta"] if kind == "chain" else 1 + case["select"] * (case["depth"] - 1)
        return dict(bytes=B * rows * case["vocab"] * (4 if case["fp32"] else 2), flops=4 * B * rows * case["vocab"])
    Hq, Hkv, d, reqs = case["q_heads"], case["kv_heads"], case["head_dim"], _requests(case)
    if kind == "verify":
        nl, row = case["layers"], 4 * Hkv * d
        # K and V of the prefix and the tree, Q, O, about two appended rows; the target's logits
        size = sum(nl * (row * (L + n) + 4 * n * Hq * d + 4 * row) + n * case["vocab"] * (4 if case["fp32"] else 2)
                   for L, n in reqs)
        return dict(bytes=size, flops=sum(nl * 4 * n * Hq * d * (L + n) for L, n in reqs))
    keys = sum(n for _, n, _, _ in reqs)              # scored keys: visual, or the whole row
    if kind == "prune":
        if case["scope"] == 0:
            keys = sum(a + n + c for a, n, c, _ in reqs)
        # rows that move, read and written (in place the rows before the image stay)
        moved = sum((0 if case["in_place"] else a) + c + r for a, _, c, r in reqs)
        return dict(bytes=keys * 2 * Hkv * d + 2 * moved * case["layers"] * 4 * Hkv * d, flops=keys * 2 * Hq * d)
    if case["guide"] == "gated":
        moved = sum(a + c + r for a, _, c, r in reqs)
        return dict(bytes=2 * keys * 2 * Hkv * d + 2 * moved * 2 * case["width"], flops=keys * 2 * Hq * d)
    rows = sum((a + n + c) * c for a, n, c, _ in reqs)
    keys = sum(a + n + c for a, n, c, _ in reqs)
    texts = sum(c for _, _, c, _ in reqs)
    return dict(bytes=keys * 2 * Hkv * d + texts * 2 * Hq * d + 4 * sum(n for _, n, _, _ in reqs), flops=rows * 2 * Hq * d)


def tolerance(case):
    if case["kind"] == "verify":
        return {"rel": 5e-3}      # bf16 inputs, probabilities and outputs, fp32 sums
    if case["kind"] == "guide" and case["guide"] == "text":
        return {"rel": 1e-3}      # probabilities cross between the stages in 16 bits
    return {"rel": 1e-5}          # fp32 sums of fp32 terms; tokens, indices and moved rows exact
