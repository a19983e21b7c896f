"""Attention of a batch whose cu_nodes run backwards, so that sequences overlap
and make more work items than the nodes alone would: the call reports the
malformed tree, and nodes that belong to one well-formed sequence only keep
their outputs, whatever place the sequence has in the order of work."""
import math

import pytest

from test_gpu_attention_ragged import _call, _inputs

pytestmark = pytest.mark.gpu


# cu_nodes, contexts, page, Hq, Hkv, D, nodes of one sequence only: the one-tile
# kernel with more items than SMs, the ping-pong kernel, and a batch small enough
# to be planned in chunks
CASES = [
    ([0, 100, 50, 150], [300, 0, 10], 0, 128, 32, 64, [(0, 0, 50), (2, 100, 150)]),
    ([0, 100, 50, 150], [300, 0, 10], 16, 256, 32, 128, [(0, 0, 50), (2, 100, 150)]),
    ([x for k in range(7) for x in (k, 128 + k)], [200] * 13, 0, 32, 8, 128,
     [(0, 0, 1), (12, 133, 134)]),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_overlapping_sequences(case):
    import torch
    from paper_2609_02897_gb300 import asd
    cu, ctx, page, Hq, Hkv, D, unique = CASES[case]
    B, T, G, cap = len(cu) - 1, cu[-1], Hq // Hkv, 512
    d = _inputs(B, 128, ctx, page, Hq, Hkv, D, cap, case)
    for k in ("q", "tree_k", "tree_v"):
        d[k] = d[k][:T].contiguous()
    parent = torch.zeros(T, dtype=torch.int32)
    parent[cu[::2]] = -1                       # every well-formed sequence is a star
    d["parent"], d["cu_nodes"] = parent.cuda(), torch.tensor(cu, dtype=torch.int32, device="cuda")
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, page, cap,
                         B * cap // page if page else 0, 128, 128)
    assert asd.asd_attention_variant(dims, T) == (3 if case == 1 else 2)
    ws = asd.alloc_workspace(dims, T)
    out = _call(d, dims, ws)
    assert asd.asd_get_device_status(ws) == 3
    for b, lo, hi in unique:
        for h in range(Hkv):
            def rows(cache):
                return (cache[d["page_table"][b].long(), h].reshape(-1, D) if page else cache[b, h])[:ctx[b]]
            for i in range(lo, hi):
                see = [cu[b]] + ([i] if i != cu[b] else [])
                k = torch.cat([rows(d["k_cache"]), d["tree_k"][see, h]]).float()
                v = torch.cat([rows(d["v_cache"]), d["tree_v"][see, h]]).float()
                x = d["q"][i, h * G:(h + 1) * G].float() @ k.T / math.sqrt(D)
                err = (out[i, h * G:(h + 1) * G].float() - x.softmax(1) @ v).abs()
                assert float(err.max()) < 2e-2, (b, i, h)   # bf16, as in the oracle comparison
