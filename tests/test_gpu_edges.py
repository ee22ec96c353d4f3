"""GPU parity at the edges of tiles, splits and slices: the sizes where a kernel's own arithmetic can go wrong."""
import numpy as np
import pytest
import torch

from oracle import twig_oracle as O
from paper_2503_14075_b200 import synth
from gpu_common import DEV, MAX_ABS_TOL, REL_L2_TOL, dev_bf16, dev_i32, f64, max_abs, rel_l2_rows
from test_gpu_chain_draft import _rows_with_top_probability
from test_gpu_tree_attn import CANARY, _wl, check, oracle_attention, run_attention
from test_gpu_tree_build import gpu_tree, gpu_tree_grown

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tw():
    from paper_2503_14075_b200 import twig
    return twig


# nodes per request, query heads per kv head, kv lengths: rows around 16, 32, 64 (instruction widths of the kernel for
# few rows) and around 128 and 256 (row blocks of the other); lengths around multiples of 8 (the tree's
# rows start on one) and of the 128-key tile
ATTN = [([1, 1, 1], 1, [0, 1, 127]), ([15, 16, 9], 1, [7, 8, 128]), ([17, 32, 31], 1, [9, 120, 129]),
        ([33, 64, 63], 1, [127, 255, 257]), ([8, 64, 1], 1, [121, 64, 383]), ([13, 5, 16], 5, [100, 385, 1023]),
        ([32, 33, 13], 4, [0, 129, 511]), ([64, 40, 37], 4, [248, 7, 640]), ([64, 37, 1], 7, [127, 256, 1025])]


@pytest.mark.parametrize("splits", [0, 1, 2, 8])
@pytest.mark.parametrize("nodes,group,kv_len", ATTN, ids=[f"rows{max(n) * g}-L{'-'.join(map(str, L))}" for n, g, L in ATTN])
def test_tcgen05_attention_tile_edges(tw, nodes, group, kv_len, splits):
    B, Hkv, d = len(nodes), 2, 128
    wl = _wl(B, Hkv * group, Hkv, d, nodes, [4] * B)
    rng = synth.rng_for(9, 811 + max(nodes) * group)
    ver = synth.make_verify_inputs(wl, rng, n_layers=1, gain=d ** 0.5)
    ck, cv = synth.make_cache(wl, rng, max(kv_len) + 67, n_layers=1, gain=d ** 0.5)
    for b in range(B):
        ck[0, b, :, kv_len[b]:] = CANARY
        cv[0, b, :, kv_len[b]:] = CANARY
    got, lse, status = run_attention(tw, wl, ver, ck, cv, kv_len, path=2, splits=splits)
    early, early_lse, early_status = run_attention(tw, wl, ver, ck, cv, kv_len, path=2, splits=splits, early=True)
    assert not status.any() and not early_status.any()
    want, want_lse = oracle_attention(ver, ck, cv, np.array(kv_len))
    check(got, lse, want, want_lse, ver["n_nodes"])
    assert np.array_equal(got, early) and np.array_equal(lse, early_lse)


@pytest.mark.parametrize("nodes,group,kv_len", ATTN[:6], ids=[f"rows{max(n) * g}" for n, g, L in ATTN[:6]])
def test_automatic_kernel_choice_head_dim_64(tw, nodes, group, kv_len):
    """A cache of 4096 keys takes the automatic choice to the tcgen05 kernel's head_dim 64 variants (more (request,
    head) pairs than SMs, and few), one of 400 to the mma.sync kernel."""
    d = 64
    for Hkv, capacity in ((2, 4096), (50, 4096), (2, 400)):
        keep = min(len(nodes), 2 if Hkv > 2 else 3)
        nn, L = nodes[:keep] + [0] * (3 - keep), [min(x, capacity - 1) for x in kv_len]
        wl = _wl(3, Hkv * group, Hkv, d, nn, [4 if x else 0 for x in nn])
        rng = synth.rng_for(9, 911 + max(nodes) * group)
        ver = synth.make_verify_inputs(wl, rng, n_layers=1, gain=d ** 0.5)
        ck, cv = (np.full((1, 3, Hkv, capacity, d), CANARY, dtype=np.uint16) for _ in range(2))
        k, v = synth.make_cache(wl, rng, max(L) + 1, n_layers=1, gain=d ** 0.5)
        for b in range(3):
            ck[0, b, :, :L[b]], cv[0, b, :, :L[b]] = k[0, b, :, :L[b]], v[0, b, :, :L[b]]
        got, lse, status = run_attention(tw, wl, ver, ck, cv, L)
        early, early_lse, _ = run_attention(tw, wl, ver, ck, cv, L, early=True)
        assert not status.any()
        want, want_lse = oracle_attention(ver, ck[:, :, :, :max(L) + 1], cv[:, :, :, :max(L) + 1], np.array(L))
        check(got, lse, want, want_lse, ver["n_nodes"])
        assert np.array_equal(got, early) and np.array_equal(lse, early_lse)


# vocabularies around the sizes at which a row is split over 2, 4 and 8 CTAs (bf16: 4096 tokens each, fp32: half)
VOCABS = [1, 8, 2047, 4096, 4103, 8191, 16385, 32769, 130001]


@pytest.mark.parametrize("fp32", [False, True], ids=["bf16", "fp32"])
@pytest.mark.parametrize("vocab", VOCABS)
def test_sliced_vocabulary_rows(tw, vocab, fp32):
    """Greedy token of a row that several CTAs share: the winner in each slice's corner, ties across slices."""
    rng = np.random.default_rng(vocab)
    T = 7
    x = rng.standard_normal((1, T, vocab)).astype(np.float32)
    for t, at in enumerate([[0], [vocab - 1], [vocab // 2], [vocab // 8, vocab - 1], [vocab // 2 - 1, vocab // 2], []]):
        for i in at:
            x[0, t, max(0, i)] = 9.0
    x[0, 6] = -np.inf                                    # everything masked: token 0
    pad = (-vocab) % 8
    if fp32:
        ref, dev = x.astype(np.float64), torch.from_numpy(np.pad(x, ((0, 0), (0, 0), (0, pad)), constant_values=3e38)).to(DEV)
    else:
        bits = synth.f32_to_bf16(x)
        ref, dev = synth.bf16_to_f64(bits), dev_bf16(np.pad(bits, ((0, 0), (0, 0), (0, pad)), constant_values=0x7F7F))
    out = torch.full((1, T), -5, dtype=torch.int32, device=DEV)
    tw.tree_base_argmax(dev[..., :vocab], dev_i32([T]), out)
    assert out.cpu().numpy()[0].tolist() == O.base_argmax(ref, [T])[0].tolist()
    # the draft step on such a row: token, probability and the early exit
    if vocab > 1:
        dx, hx = _rows_with_top_probability(rng, 2, vocab, [0.9, 0.3], fp32)
        d2 = torch.from_numpy(np.pad(dx, ((0, 0), (0, pad)))).to(DEV) if fp32 else dev_bf16(np.pad(dx, ((0, 0), (0, pad))))
        par, tok = (torch.full((2, 4), -7, dtype=torch.int32, device=DEV) for _ in range(2))
        n, active = (torch.full((2,), -7, dtype=torch.int32, device=DEV) for _ in range(2))
        prob = torch.full((2, 4), -7.0, dtype=torch.float32, device=DEV)
        tw.chain_draft_reset(par, tok, n, active, tok_prob=prob)
        tw.chain_draft_step(d2[:, :vocab], 3, 0.6, par, tok, n, active, tok_prob=prob)
        for b in range(2):
            want_t, want_p = O.chain_draft([hx[b]], 3, 0.6)
            assert tok.cpu().numpy()[b, 1] == want_t[0] and np.allclose(prob.cpu().numpy()[b, 1], want_p[0], rtol=2e-4)
        assert active.cpu().tolist() == [1, 0]


@pytest.mark.parametrize("grown", [False, True], ids=["calls", "one-launch-per-level"])
@pytest.mark.parametrize("E,K,D,n_max,V,B", [(16, 16, 4, 64, 8191, 2), (16, 16, 6, 64, 4103, 1), (2, 1, 6, 8, 16385, 1), (16, 3, 2, 40, 131, 40)])
def test_tree_levels_over_slices(tw, E, K, D, n_max, V, B, grown):
    """Rows split over a cluster (few requests) and not (many), trees of more nodes than a CTA has threads,
    scores tied at the selection's boundary (two requests of equal rows)."""
    rng = synth.rng_for(7, 90 + V % 50)
    host, dev = [], []
    for l in range(D):
        x = (rng.standard_normal((B, 1 if l == 0 else K, V)) * 3.0).astype(np.float32)
        x[-1, :, 1::2] = x[-1, :, 0:V - 1:2]              # the last request: every logit twice
        host.append(x.astype(np.float64))
        dev.append(torch.from_numpy(np.pad(x, ((0, 0), (0, 0), (0, (-V) % 8)))).to(DEV)[..., :V])
    parent, tok, n_nodes, kept, status, _ = (gpu_tree_grown if grown else gpu_tree)(tw, dev, E, K, n_max, 64)
    assert not status.any()
    for b in range(B):
        p_o, t_o, _, keep_o, _ = O.build_token_tree([h[b] for h in host], E, K, n_max)
        n = len(p_o)
        assert n_nodes[b] == n and np.array_equal(kept[b, :n], keep_o)
        assert np.array_equal(parent[b, :n], p_o) and np.array_equal(tok[b, :n], t_o)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens", [[(0, 64, 0), (1, 62, 0)], [(63, 1, 0), (64, 65, 1)], [(5, 4097, 63), (0, 1, 0)],
                                  [(7, 511, 2), (0, 513, 1), (130, 1024, 500)]], ids=lambda x: f"{len(x)}-{x[0][1]}")
def test_score_chunk_edges(tw, lens, d):
    """Scores with and without gates at the edges of the 64-key chunks, and more tokens than the selection has threads."""
    B, Hq, Hkv = len(lens), 6, 3
    before, n_vis, after = (np.array([x[i] for x in lens], dtype=np.int32) for i in range(3))
    total = before + n_vis + after
    rng = synth.rng_for(9, int(total.max()))
    q, qg = (synth.normal_bf16(rng, (B, Hq, d), d, d ** 0.5) for _ in range(2))
    k, kg = (synth.normal_bf16(rng, (B, Hkv, int(total.max()) + 3, d), d, d ** 0.5) for _ in range(2))
    for b in range(B):
        k[b, :, total[b]:] = CANARY                       # NaN past the prompt
        kg[b, :, total[b]:] = CANARY
    clean = [np.where(np.arange(x.shape[2])[None, None, :, None] < total[:, None, None, None], x, 0) for x in (k, kg)]
    ws = torch.empty(tw.twig_workspace_bytes(B, Hq, d, k.shape[2], 64), dtype=torch.uint8, device=DEV)
    args = (dev_i32(total), dev_i32(before), dev_i32(n_vis))
    for scope in (0, 1):
        got = torch.full((B, int(n_vis.max())), -1.0, dtype=torch.float32, device=DEV)
        gated, status = torch.full_like(got, -1.0), torch.zeros(B, dtype=torch.int32, device=DEV)
        tw.ttp_score(dev_bf16(q), dev_bf16(k), *args, got, ws, norm_scope=scope, dev_status=status)
        tw.ttp_score_gated(dev_bf16(q), dev_bf16(qg), dev_bf16(k), dev_bf16(kg), *args, gated, ws, norm_scope=scope, dev_status=status)
        assert not status.any()
        want = O.ttp_scores(f64(q), f64(clean[0]), total, before, n_vis, scope)
        want_g = O.ttp_scores_gated(f64(q), f64(qg), f64(clean[0]), f64(clean[1]), total, before, n_vis, scope)
        for have, ref in ((got.cpu().numpy(), want), (gated.cpu().numpy(), want_g)):
            for b in range(B):
                assert max_abs(have[b, :n_vis[b]], ref[b][:n_vis[b]]) <= 1e-4
                assert rel_l2_rows(have[b, :n_vis[b]].astype(np.float64), ref[b][:n_vis[b]]) <= REL_L2_TOL


# (visual tokens, text tokens, kv heads, head_dim): chunks of 128 keys and shares of a cluster of 1 to 8 CTAs; 4096 keys is
# the last length of the one-pass kernel; 64 text rows are a block
MULTI = [(1, 1, 1, 64), (63, 65, 2, 128), (511, 64, 2, 128), (3968, 120, 1, 128), (4030, 63, 1, 64), (4090, 70, 1, 128), (900, 130, 16, 64)]


@pytest.mark.parametrize("n_vis,n_text,Hkv,d", MULTI)
def test_multiquery_kernel_edges(tw, n_vis, n_text, Hkv, d):
    B, Hq = 2, Hkv * 2
    before = np.array([3, 0], dtype=np.int32)
    vis = np.array([n_vis, max(1, n_vis // 3)], dtype=np.int32)
    text = np.array([n_text, max(1, n_text - 1)], dtype=np.int32)
    total = before + vis + text
    rng = synth.rng_for(9, n_vis + n_text)
    k = synth.normal_bf16(rng, (B, Hkv, int(total.max()), d), d, d ** 0.5)
    q = synth.normal_bf16(rng, (B, Hq, n_text, d), d, d ** 0.5)
    k[:, 0, 5::17] = synth.f32_to_bf16(8.0 * synth.bf16_to_f64(k[:, 0, 5::17]).astype(np.float32))      # logits that raise a row's reference
    scores = torch.full((B, n_vis), -1.0, dtype=torch.float32, device=DEV)
    ws = torch.empty(tw.ttp_multiquery_workspace_bytes(B, Hq, n_text, n_vis, k.shape[2]), dtype=torch.uint8, device=DEV)
    status = torch.zeros(B, dtype=torch.int32, device=DEV)
    tw.ttp_score_multiquery(dev_bf16(q), dev_bf16(k), dev_i32(total), dev_i32(before), dev_i32(vis), scores, ws, dev_status=status)
    got = scores.cpu().numpy()
    assert not status.any()
    want = O.text_to_visual_scores(f64(q), f64(k), total, before, vis)
    for b in range(B):
        assert max_abs(got[b, :vis[b]], want[b][:vis[b]]) <= MAX_ABS_TOL
        assert rel_l2_rows(got[b, :vis[b]].astype(np.float64), want[b][:vis[b]]) <= REL_L2_TOL
        assert np.all(got[b, vis[b]:] == 0)
