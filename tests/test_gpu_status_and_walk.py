"""Calls of the short kernels at the batch sizes where their launch changes: the
walk and the commit as one cluster that clears the status word (up to 16
sequences; beyond 8 not a portable cluster size) or behind a kernel that does,
and the tree preparation in one CTA (up to 32 sequences, eight at a time) or
several.  The walk under every accept rule against the oracle; the status word
is clean after a call on good inputs that follows one on bad inputs, and a
malformed tree in any position is reported and does not touch the others."""
import numpy as np
import pytest

import oracle
from paper_2609_02897_gb300 import synth

pytestmark = pytest.mark.gpu


def _batch(B, seed, vocab=50):
    rng = np.random.default_rng(seed)
    trees = [synth.random_topological_relabel(
        synth.tree_grown(rng, int(rng.integers(1, 129)), int(rng.integers(1, 13)),
                         int(rng.integers(1, 17))), rng) for _ in range(B)]
    cu = np.concatenate([[0], np.cumsum([len(t) for t in trees])]).astype(np.int32)
    T = int(cu[-1])
    parent = np.concatenate(trees).astype(np.int32)
    accept = (rng.random(T) < 0.75).astype(np.uint8)
    arg = rng.integers(0, vocab, T).astype(np.int32)
    tokens = rng.integers(0, vocab, T).astype(np.int32)
    for b in range(B):
        for i in range(cu[b] + 1, cu[b + 1]):
            if accept[i] and rng.random() < 0.5:
                tokens[i] = arg[cu[b] + parent[i]]          # a strict match
    ratio = rng.integers(1, 6, T).astype(np.float32) / 8    # ties among siblings
    return parent, tokens, accept, arg, ratio, cu


@pytest.mark.parametrize("B", [1, 2, 7, 8, 9, 16, 17, 33])
@pytest.mark.parametrize("rule", [0, 1, 2, 3])
def test_walk_and_commit(B, rule):
    import torch
    from paper_2609_02897_gb300 import asd
    parent, tokens, accept, arg, ratio, cu = _batch(B, 10 * B + rule)
    T, Hkv, D, cap, max_path = int(cu[-1]), 2, 64, 64, 16
    dims = asd.make_dims(B, 2, Hkv, D, 64, 50, asd.ASD_BF16, 0, cap, 0, 128, max_path, accept_rule=rule)
    ws = asd.alloc_workspace(dims, T)
    dev = {k: torch.from_numpy(v).cuda() for k, v in dict(
        parent=parent, tokens=tokens, accept=accept, arg=arg, ratio=ratio, cu=cu).items()}
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")  # noqa: E731
    path, plen, bonus, npro, cout = i32(B, max_path), i32(B), i32(B), i32(B), i32(B)
    ctx = torch.arange(B, dtype=torch.int32, device="cuda") % 7
    tk, tv = (torch.randn(T, Hkv, D, device="cuda").to(torch.bfloat16) for _ in range(2))
    kc, vc = (torch.zeros(B, Hkv, cap, D, dtype=torch.bfloat16, device="cuda") for _ in range(2))

    def walk(par):
        asd.asd_accept_path(dims, par, dev["tokens"], dev["accept"], dev["arg"], dev["cu"], path, plen,
                            bonus, npro, ws, ratio=dev["ratio"])

    def commit():
        asd.asd_kv_compact(dims, tk, tv, dev["cu"], T, path, plen, ctx, None, kc, vc, cout, ws)

    bad = dev["parent"].clone()
    bad[int(cu[B - 1])] = 5                      # the last sequence's root has a parent
    walk(bad)
    assert asd.asd_get_device_status(ws) == 3
    assert int(plen[B - 1]) == 0 and (B == 1 or int(plen[0]) > 0)
    walk(dev["parent"])
    assert asd.asd_get_device_status(ws) == 0
    want, wlen, wbonus, wpro = oracle.accept_path(parent, accept, arg, tokens, cu, rule=rule, ratio=ratio)
    assert plen.tolist() == list(wlen) and bonus.tolist() == list(wbonus)
    assert npro.tolist() == list(wpro)
    got = path.cpu().numpy()
    for b in range(B):
        assert got[b][:len(want[b])].tolist() == list(want[b]) and np.all(got[b][len(want[b]):] == -1)
    commit()
    assert asd.asd_get_device_status(ws) == 0
    assert cout.tolist() == [int(c) + len(w) for c, w in zip(ctx.tolist(), want)]
    for b in range(B):
        rows = torch.tensor([int(cu[b]) + u for u in want[b]], device="cuda")
        c0 = int(ctx[b])
        for cache, tree in ((kc, tk), (vc, tv)):
            assert torch.equal(cache[b, :, c0:c0 + len(rows)], tree[rows].transpose(0, 1))
            assert float(cache[b, :, c0 + len(rows):].abs().sum()) == 0 and \
                float(cache[b, :, :c0].abs().sum()) == 0
    plen[B - 1] = 999                            # longer than max_path
    commit()
    assert asd.asd_get_device_status(ws) == 2
    assert int(cout[B - 1]) == int(ctx[B - 1])


@pytest.mark.parametrize("B", [8, 9, 16, 17])
def test_walk_and_commit_in_a_captured_graph(B):
    """The cluster launches, the non-portable sizes among them, and the kernel that
    clears the status word beyond 16 sequences, recorded and replayed on other
    inputs in the same buffers."""
    import torch
    from paper_2609_02897_gb300 import asd
    first = _batch(B, 100 + B)
    parent, _, _, _, _, cu = first
    rng = np.random.default_rng(B)
    T, Hkv, D, cap, max_path = int(cu[-1]), 2, 64, 64, 16
    # the same trees, other verdicts
    second = (parent, rng.integers(0, 50, T).astype(np.int32), (rng.random(T) < 0.6).astype(np.uint8),
              rng.integers(0, 50, T).astype(np.int32), first[4], cu)
    dims = asd.make_dims(B, 2, Hkv, D, 64, 50, asd.ASD_BF16, 0, cap, 0, 128, max_path)
    ws = asd.alloc_workspace(dims, T)
    dev = [torch.from_numpy(x.copy()).cuda() for x in first]
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device="cuda")  # noqa: E731
    path, plen, bonus, npro, cout, ctx = i32(B, max_path), i32(B), i32(B), i32(B), i32(B), i32(B)
    tk, tv = (torch.randn(T, Hkv, D, device="cuda").to(torch.bfloat16) for _ in range(2))
    kc, vc = (torch.zeros(B, Hkv, cap, D, dtype=torch.bfloat16, device="cuda") for _ in range(2))

    def calls():
        asd.asd_accept_path(dims, dev[0], dev[1], dev[2], dev[3], dev[5], path, plen, bonus, npro, ws,
                            ratio=dev[4])
        asd.asd_kv_compact(dims, tk, tv, dev[5], T, path, plen, ctx, None, kc, vc, cout, ws)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for batch in (first, second):
        for t, x in zip(dev, batch):
            t.copy_(torch.from_numpy(x.copy()))
        kc.zero_()
        graph.replay()
        assert asd.asd_get_device_status(ws) == 0
        want, wlen, wbonus, _ = oracle.accept_path(parent, batch[2], batch[3], batch[1], cu, rule=0,
                                                   ratio=batch[4])
        assert plen.tolist() == list(wlen) and bonus.tolist() == list(wbonus) and cout.tolist() == list(wlen)
        for b in range(B):
            rows = torch.tensor([int(cu[b]) + u for u in want[b]], device="cuda")
            assert torch.equal(kc[b, :, :len(rows)], tk[rows].transpose(0, 1))


@pytest.mark.parametrize("B", [1, 8, 9, 32, 33, 40])
def test_tree_preparation_reports_any_sequence(B):
    import torch
    from paper_2609_02897_gb300 import asd
    n, V, K = 5, 300, 64
    T = B * n
    dims = asd.make_dims(B, 2, 2, 64, K, V, asd.ASD_BF16, 0, 64, 0, n, n)
    g = torch.Generator(device="cuda").manual_seed(B)
    h = torch.randn(T, K, generator=g, device="cuda").to(torch.bfloat16)
    w = torch.randn(V, K, generator=g, device="cuda").to(torch.bfloat16)
    tokens = torch.randint(0, V, (T,), generator=g, device="cuda").int()
    parent = torch.tensor([-1, 0, 0, 1, 1], dtype=torch.int32).repeat(B).cuda()
    cu = torch.arange(0, T + 1, n, dtype=torch.int32, device="cuda")
    ws = asd.alloc_workspace(dims, T)
    out = {k: torch.zeros(T, dtype=torch.float32, device="cuda")
           for k in ("row_max", "row_lse", "l_draft", "ratio")}
    out["row_argmax"] = torch.zeros(T, dtype=torch.int32, device="cuda")
    out["accept"] = torch.zeros(T, dtype=torch.uint8, device="cuda")

    def call(par, tok):
        asd.asd_lmhead_margin(dims, h, w, tok, par, cu, 0.5, workspace=ws, **out)
        return asd.asd_get_device_status(ws)

    assert call(parent, tokens) == 0
    good = {k: v.clone() for k, v in out.items()}
    ref = h.float() @ w.float().T
    gp = torch.arange(T, device="cuda") // n * n + parent.long()
    kids = parent >= 0
    # sums of 64 products of bf16 values in fp32: 2^-18 of their magnitude
    want = ref[gp[kids], tokens[kids].long()]
    assert float((good["l_draft"][kids] - want).abs().max()) < 64 * 2.0 ** -14
    for b in sorted({0, B // 2, B - 1}):
        bad = parent.clone()
        bad[b * n + 3] = 4                       # a parent behind its child
        assert call(bad, tokens) == 3
        tok = tokens.clone()
        tok[b * n + 2] = V
        assert call(parent, tok) == 4
        assert call(parent, tokens) == 0
        for k, v in out.items():
            assert torch.equal(v.view(torch.uint8), good[k].view(torch.uint8)), k
