"""Tree attention over ragged context lengths on full-size caches, with more
work items than SMs, against a plain PyTorch fp32 reference, and repeated: a
context that ends inside a 128-key tile has its tail V rows zeroed in shared
memory, which must wait for the V ring however late it runs (it runs late when
other CTAs start their first copies)."""
import math

import pytest

pytestmark = pytest.mark.gpu


def _inputs(B, n, ctx, page, Hq, Hkv, D, cap, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)

    T = B * n
    d = dict(q=normal(T, Hq, D), tree_k=normal(T, Hkv, D), tree_v=normal(T, Hkv, D))
    if page:
        per = cap // page
        d["k_cache"], d["v_cache"] = (normal(B * per, Hkv, page, D) for _ in range(2))
        d["page_table"] = torch.randperm(B * per, generator=g, device="cuda").view(B, per).int()
    else:
        d["k_cache"], d["v_cache"] = (normal(B, Hkv, cap, D) for _ in range(2))
        d["page_table"] = None
    d["ctx_len"] = torch.tensor(ctx, dtype=torch.int32, device="cuda")
    # a binary tree: parent of node i is (i - 1) // 2
    par = torch.tensor([(i - 1) // 2 if i else -1 for i in range(n)], dtype=torch.int32)
    d["parent"] = par.repeat(B).cuda()
    d["cu_nodes"] = torch.arange(0, T + 1, n, dtype=torch.int32, device="cuda")
    return d


def _reference(d, B, n, ctx, page, Hq, Hkv, D):
    """fp32 softmax attention of every node over its context and ancestors."""
    import torch
    G = Hq // Hkv
    see = torch.eye(n, dtype=torch.bool)
    for i in range(1, n):
        see[i] |= see[(i - 1) // 2]
    hide = ~see.cuda().repeat_interleave(G, 0)
    out = torch.empty(B * n, Hq, D, device="cuda")
    for b in range(B):
        for h in range(Hkv):
            def keys(cache, tree):
                rows = (cache[d["page_table"][b].long(), h].reshape(-1, D) if page else cache[b, h])
                return torch.cat([rows[:ctx[b]], tree[b * n:(b + 1) * n, h]]).float()
            q = d["q"][b * n:(b + 1) * n, h * G:(h + 1) * G].reshape(n * G, D).float()
            x = q @ keys(d["k_cache"], d["tree_k"]).T / math.sqrt(D)
            x[:, ctx[b]:].masked_fill_(hide, -math.inf)
            out[b * n:(b + 1) * n, h * G:(h + 1) * G] = \
                (x.softmax(1) @ keys(d["v_cache"], d["tree_v"])).view(n, G, D)
    return out


def _call(d, dims, ws):
    import torch
    from paper_2609_02897_gb300 import asd
    out = torch.full_like(d["q"], float("nan"))
    asd.asd_tree_attention(dims, d["q"], d["k_cache"], d["v_cache"], d["page_table"], d["ctx_len"],
                           d["tree_k"], d["tree_v"], d["parent"], d["cu_nodes"], out, ws)
    return out


def _check_close(out, ref):
    # bf16 outputs from bf16 probabilities (8 significant bits each): every
    # output is a mean of N(0, 1) values, and 2e-2 absolute is the tolerance of
    # the oracle comparison; the mean error is far below it
    err = (out.float() - ref).abs()
    assert bool((err <= 2e-2 + 1e-2 * ref.abs()).all()), float(err.max())
    assert float((out.float() - ref).norm() / ref.norm()) < 5e-3


@pytest.mark.parametrize("D,page", [(128, 0), (128, 16), (64, 0)])
def test_late_v_ring_does_not_disturb_a_ragged_tail(D, page):
    import torch
    from paper_2609_02897_gb300 import asd
    B, n, Hq, Hkv, cap = 32, 6, 32, 8, 8192
    ctx = [1024 + (b * 2741) % 7160 + (b % 127) for b in range(B)]   # 1024 .. 8190, ragged
    d = _inputs(B, n, ctx, page, Hq, Hkv, D, cap, 3)
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, page, cap,
                         B * cap // page if page else 0, n, n)
    ws = asd.alloc_workspace(dims, B * n)
    outs = [_call(d, dims, ws) for _ in range(60)]
    assert asd.asd_get_device_status(ws) == 0
    _check_close(outs[0], _reference(d, B, n, ctx, page, Hq, Hkv, D))
    for o in outs[1:]:
        assert torch.equal(o.view(torch.int16), outs[0].view(torch.int16))


# (B, nodes, contexts, page, Hq, Hkv, D, cache slots): chunk and tile edges, a
# cache much larger than the contexts, ragged batches in which only the long
# sequences are cut, more than 128 nodes, query groups that do not divide 128
SPLITS = [
    (1, 1, [0], 0, 32, 8, 128, 4096),
    (1, 8, [127], 0, 32, 8, 128, 40960),
    (1, 8, [128], 16, 32, 8, 128, 4096),
    (1, 8, [129], 0, 32, 8, 64, 4096),
    (1, 5, [4095], 0, 32, 8, 128, 32768),
    (1, 60, [2049], 0, 32, 8, 128, 2112),
    (1, 128, [9000], 64, 16, 8, 128, 16384),
    (3, 7, [0, 257, 6001], 16, 28, 4, 128, 8192),
    (4, 33, [511, 4000, 130, 2600], 256, 32, 8, 128, 8192),
    (2, 100, [3000, 700], 0, 64, 8, 64, 4096),
    (19, 6, [100 * (b + 1) + b for b in range(19)], 8, 8, 1, 128, 2048),
]


@pytest.mark.parametrize("case", range(len(SPLITS)))
@pytest.mark.parametrize("small_workspace", [False, True])
def test_split_contexts(case, small_workspace):
    """Contexts cut into chunks and merged, and the same call with a workspace
    that ends before (most of) the partial rows, which splits less."""
    import torch
    from paper_2609_02897_gb300 import asd
    B, n, ctx, page, Hq, Hkv, D, cap = SPLITS[case]
    d = _inputs(B, n, ctx, page, Hq, Hkv, D, cap, case)
    # one vocabulary range: the workspace before the partial rows is small
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 32, asd.ASD_BF16, page, cap,
                         B * cap // page if page else 0, n, n)
    ws = asd.alloc_workspace(dims, B * n)
    if small_workspace:
        ws = ws[:min(ws.numel(), 32768)]
    out = _call(d, dims, ws)
    again = _call(d, dims, ws)
    assert asd.asd_get_device_status(ws) == 0
    _check_close(out, _reference(d, B, n, ctx, page, Hq, Hkv, D))
    assert torch.equal(out.view(torch.int16), again.view(torch.int16))


def test_split_batch_with_a_malformed_sequence():
    """A malformed sequence in a batch that splits gets no work and is
    reported; the others' outputs are those of the batch without the fault, up
    to the rounding of another cut (the chunk length follows the whole batch)."""
    from paper_2609_02897_gb300 import asd
    B, n, Hq, Hkv, D, cap = 3, 8, 32, 8, 128, 8192
    d = _inputs(B, n, [5000, 3000, 7000], 0, Hq, Hkv, D, cap, 1)
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 32, asd.ASD_BF16, 0, cap, 0, n, n)
    ws = asd.alloc_workspace(dims, B * n)
    good = _call(d, dims, ws)
    assert asd.asd_get_device_status(ws) == 0
    d["cu_nodes"][2] = d["cu_nodes"][1]          # sequence 1 empty, 2 too long
    out = _call(d, dims, ws)
    assert asd.asd_get_device_status(ws) == 3
    _check_close(out[:n], good[:n].float())


# contexts short enough for the kernel beside the LM head and too long for it,
# in the same cache of 24576 slots (small LM head: the limit is 16 key tiles of
# 32 keys on the busiest SM)
@pytest.mark.parametrize("ctx", [[0, 5], [300, 1500], [20000, 40], [24000, 23999], [1, 24500]])
@pytest.mark.parametrize("D,page,nodes", [(128, 0, 40), (64, 16, 9)])
@pytest.mark.parametrize("lazy", [False, True])
def test_small_steps_choose_their_attention_by_context(ctx, D, page, nodes, lazy):
    import torch
    from paper_2609_02897_gb300 import asd
    B, Hq, Hkv, cap, hidden, vocab = 2, 16, 4, 24576, 64, 200
    d = _inputs(B, nodes, ctx, page, Hq, Hkv, D, cap, 7)
    g = torch.Generator(device="cuda").manual_seed(9)
    d["hidden"] = torch.randn(B * nodes, hidden, generator=g, device="cuda").to(torch.bfloat16)
    d["w_lm"] = torch.randn(vocab, hidden, generator=g, device="cuda").to(torch.bfloat16)
    d["tokens"] = torch.randint(0, vocab, (B * nodes,), generator=g, device="cuda").int()
    dims = asd.make_dims(B, Hq, Hkv, D, hidden, vocab, asd.ASD_BF16, page, cap,
                         B * cap // page if page else 0, nodes, 8,
                         lm_head_schedule=1 if lazy else 0)
    step = asd.VerifyStep(dims, B * nodes).bind(tau=0.5, **d)
    ref = _reference(d, B, nodes, ctx, page, Hq, Hkv, D)
    for _ in range(2):
        step.out["attn_out"].fill_(float("nan"))
        out = step.run()["attn_out"]
        assert step.device_status() == 0
        _check_close(out, ref)
