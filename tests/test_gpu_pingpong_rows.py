"""The ping-pong attention's two query tiles at the row counts where they
change (one tile only, a full first tile, one row in the second, both full) in
one ragged batch, against a plain PyTorch fp32 reference, with several waves of
items and with about one.  Keys grow along the context, so that the running
maximum is raised, and O rescaled, more than once.  And which form a call takes
on both sides of every line of the rule."""
import pytest

from test_gpu_attention_ragged import _call, _check_close, _inputs, _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,page,Hq", [(64, 128, 0, 32), (64, 128, 16, 32), (64, 64, 0, 32),
                                         (64, 64, 64, 24), (24, 128, 16, 32), (32, 64, 0, 32)])
def test_row_counts_of_the_two_query_tiles(B, D, page, Hq):
    import torch
    from paper_2609_02897_gb300 import asd
    Hkv, N, cap = 8, 128, 1024
    nodes = [(1, 31, 32, 33, 43, 64, 127, 128)[b % 8] for b in range(B)]
    ctx = [(0, 1, 127, 128, 129, 300, 640, 895)[(b // 8 + b) % 8] for b in range(B)]
    full = _inputs(B, N, ctx, page, Hq, Hkv, D, cap, 5)
    # a score's standard deviation rises from 1 to 8 over the cache
    if page == 0:
        full["k_cache"] *= torch.linspace(1, 8, cap, device="cuda").view(1, 1, cap, 1)
    else:
        of_page = torch.empty(B * cap // page, device="cuda")
        of_page[full["page_table"].long()] = torch.linspace(1, 8, cap // page, device="cuda")
        full["k_cache"] *= of_page.view(-1, 1, 1, 1)
    # each sequence keeps its first nodes (a prefix of the binary tree is one)
    rows = torch.cat([torch.arange(b * N, b * N + n) for b, n in enumerate(nodes)]).cuda()
    d = dict(full)
    for k in ("q", "tree_k", "tree_v", "parent"):
        d[k] = full[k][rows].contiguous()
    d["cu_nodes"] = torch.tensor([0] + nodes).cumsum(0).int().cuda()
    T = sum(nodes)
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, page, cap,
                         B * cap // page if page else 0, N, N)
    assert asd.asd_attention_variant(dims, T) == 3
    out = _call(d, dims, asd.alloc_workspace(dims, T))
    s = 0
    for b, n in enumerate(nodes):
        one = {k: d[k][s:s + n] for k in ("q", "tree_k", "tree_v")}
        one["page_table"] = d["page_table"][b:b + 1] if page else None
        for k in ("k_cache", "v_cache"):
            one[k] = d[k] if page else d[k][b:b + 1]
        _check_close(out[s:s + n], _reference(one, 1, n, ctx[b:b + 1], page, Hq, Hkv, D))
        s += n


def test_which_form_a_call_takes():
    import torch
    from paper_2609_02897_gb300 import asd
    nsm = torch.cuda.get_device_properties(0).multi_processor_count

    def form(items, page=0, batch=1):
        # one KV head and G = 2: an item is 128 nodes
        dims = asd.make_dims(max(batch, items), 2, 1, 128, 64, 64, asd.ASD_BF16, page, 1024,
                             64 if page else 0, 128, 8)
        return asd.asd_attention_variant(dims, 128 * items)

    low, half = -(-5 * nsm // 6), 3 * nsm // 2
    assert [form(low - 1), form(low), form(nsm), form(nsm + 1), form(half), form(half + 1)] == \
        [2, 3, 3, 2, 2, 3]
    assert [form(low - 1, 16), form(nsm + 1, 32), form(half, 16), form(half, 64)] == [2, 3, 3, 2]
    # 128 rows per sequence on average: the second query tile would stay empty
    assert form(4 * nsm) == 3 and form(4 * nsm, batch=8 * nsm) == 2

    def of_nodes(n, batch, G):
        dims = asd.make_dims(batch, G, 1, 128, 64, 64, asd.ASD_BF16, 0, 1024, 0, 128, 8)
        return asd.asd_attention_variant(dims, n * batch)

    # 100 nodes of G = 3 are 300 rows: three tiles, but two pairs, the second half
    # empty; from two waves of all rows on pairs whatever the sizes
    assert [of_nodes(100, 7 * nsm * 256 // 4 // 300, 3), of_nodes(100, 2 * nsm, 3)] == [2, 3]


def test_about_one_wave_of_pairs_the_contexts_decide():
    """Equal contexts run the two-tile form, a batch whose longest context stands
    out single tiles, at both sides of the line; told by the bits of the same
    sequences in a batch of fewer (single tiles) and of more (pairs)."""
    import torch
    from paper_2609_02897_gb300 import asd
    Hq, Hkv, D, n, cap = 32, 8, 128, 128, 4096
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    mid, few, many = nsm // 16, 5 * nsm // 6 // 16 - 1, 3 * nsm // 2 // 16 + 1   # 16 pairs each
    g = 1024 // 128 + 1              # key tiles of the others, the tree's among them
    # the longest, t tiles: t <= 0.56 max(t, 1.15 work / nsm) + 3, 32 items each
    line = max(t for t in range(g, 33)
               if t <= 0.56 * max(t, 1.15 * 32 * (t + g * (mid - 1)) / nsm) + 3)
    assert g < line < 32

    def run(B, ctx):
        d = dict(full, ctx_len=torch.tensor(ctx, dtype=torch.int32, device="cuda"))
        for k in ("q", "tree_k", "tree_v", "parent"):
            d[k] = full[k][:B * n].contiguous()
        for k in ("k_cache", "v_cache"):
            d[k] = full[k][:B].contiguous()
        d["cu_nodes"] = torch.arange(0, B * n + 1, n, dtype=torch.int32, device="cuda")
        dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, 0, cap, 0, n, n)
        assert asd.asd_attention_variant(dims, B * n) == (2 if B == few else 3)
        return _call(d, dims, asd.alloc_workspace(dims, B * n))[:few * n].view(torch.int16)

    full = _inputs(many, n, [0] * many, 0, Hq, Hkv, D, cap, 3)
    for longest, pairs in ((g, True), (line, True), (line + 1, False), (32, False)):
        ctx = [1024] * many
        ctx[1] = 128 * (longest - 1)
        out, single, double = run(mid, ctx[:mid]), run(few, ctx[:few]), run(many, ctx)
        assert not torch.equal(single, double)
        assert torch.equal(out, double if pairs else single), (longest, pairs)
