"""The exact fp32 kernels over their tile edges, against the fp64 oracle: node
tiles of 8, 16, 32 and 64 with ragged ends, hidden widths that are not a
multiple of 4 (rows then start unaligned), vocabularies that end inside a chunk
and a range, 64-row query blocks, both head sizes, query groups, paged caches,
empty and short contexts."""
import numpy as np
import pytest

import _helpers as H
from paper_2609_02897_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import _device
    return _device


@pytest.mark.parametrize("over", [
    dict(B=1, nodes=1, ctx=(0, 0), hidden=1, vocab=7),
    dict(B=1, nodes=8, ctx=(31, 31), hidden=257, vocab=4097),
    dict(B=3, nodes=3, ctx=(1, 33), hidden=100, vocab=1000, page_size=16),
    dict(B=2, nodes=9, ctx=(200, 400), hidden=64, vocab=9733, D=128, Hq=8, Hkv=4),
    dict(B=4, nodes=8, ctx=(64, 65), hidden=63, vocab=511, D=128, page_size=8),
    dict(B=3, nodes=21, ctx=(0, 90), hidden=260, vocab=300, Hq=6, Hkv=2),
    dict(B=2, nodes=128, ctx=(600, 700), hidden=132, vocab=1201, Hq=8, Hkv=2, page_size=256),
])
def test_f32_tile_edges(dev, over):
    over = dict(over)
    B, n = over["B"], over.pop("nodes")
    rng = np.random.default_rng(n)
    trees = [synth.tree_grown(rng, n, 1 + b % 6, 1 + b % 4 if n < 10 else 40) for b in range(B)]
    wl = H.prepared(1, overrides=over, tree_override=trees)
    for tau in (1.0, 0.3):
        out, status, _, _ = dev.run_verify(wl, tau)
        assert status == 0
        H.compare_verify(wl, tau, out)
        H.untouched_cache_equal(wl, out, [(b, int(wl.ctx_len[b]) + k) for b in range(B)
                                          for k in range(int(out["path_len"][b]))])


def test_f32_masked_value_rows_may_hold_anything(dev):
    """A drafted node's V row is read by its descendants only: NaN in one
    branch stays out of the others."""
    import torch
    from paper_2609_02897_gb300 import asd
    wl = H.prepared(1, tree_override=[np.array([-1, 0, 0, 1, 2], dtype=np.int32)])
    d = dev.to_device(wl)
    dims = dev.dims_of(wl)
    ws = asd.alloc_workspace(dims, wl.T)
    outs = []
    for poison in (False, True):
        if poison:
            d["tree_v"][1] = float("nan")
        out = torch.empty_like(d["q"])
        asd.asd_tree_attention(dims, d["q"], d["k_cache"], d["v_cache"], d["page_table"], d["ctx_len"],
                               d["tree_k"], d["tree_v"], d["parent"], d["cu_nodes"], out, ws)
        outs.append(out)
    keep = [0, 2, 4]      # neither node 1 nor its child 3
    assert torch.equal(outs[0][keep], outs[1][keep])
    assert bool(torch.isnan(outs[1][[1, 3]]).all())
