"""Precision of the tensor-core attention in calls of up to 128 nodes, against
64 bits.  Rounding to bf16 numbers whose leading bits are spread evenly over an
octave is an error of u = 2^-7 / sqrt(12) * sqrt((1 - 2^-2) / (2 ln 2)) = 1.66e-3
in the 2-norm.  The output is rounded once; of P, half the weights are (the
other half goes to the P.V product in two bf16 terms), and V being independent
their errors add in squares: sqrt(u^2 + u^2 / 2) = 2.03e-3, less where the
largest weights are powers of two.  The bound leaves 2 % for the sample; all of
P in one term gives 2.1e-3 to 2.35e-3."""
import math

import pytest

from test_gpu_attention_ragged import _call, _inputs

pytestmark = pytest.mark.gpu

BOUND = 2.07e-3


def _exact(d, B, n, ctx, page, Hq, Hkv, D):
    import torch
    G = Hq // Hkv
    see = torch.eye(n, dtype=torch.bool)
    for i in range(1, n):
        see[i] |= see[(i - 1) // 2]
    hide = ~see.cuda().repeat_interleave(G, 0)
    out = torch.empty(B * n, Hq, D, dtype=torch.float64, device="cuda")
    for b in range(B):
        for h in range(Hkv):
            def keys(cache, tree):
                rows = (cache[d["page_table"][b].long(), h].reshape(-1, D) if page else cache[b, h])
                return torch.cat([rows[:ctx[b]], tree[b * n:(b + 1) * n, h]]).double()
            q = d["q"][b * n:(b + 1) * n, h * G:(h + 1) * G].reshape(n * G, D).double()
            x = q @ keys(d["k_cache"], d["tree_k"]).T / math.sqrt(D)
            x[:, ctx[b]:].masked_fill_(hide, -math.inf)
            out[b * n:(b + 1) * n, h * G:(h + 1) * G] = \
                (x.softmax(1) @ keys(d["v_cache"], d["tree_v"])).view(n, G, D)
    return out


# (B, nodes, contexts, page, D): one chunk and several, one key tile and many,
# a running maximum that is raised more than once (32768 keys)
CASES = [
    (1, 8, [500], 0, 128),
    (1, 128, [500], 0, 128),
    (2, 60, [300, 2048], 16, 128),
    (4, 32, [100, 4000, 130, 2600], 0, 64),
    (1, 8, [32768], 0, 128),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_calls_of_up_to_128_nodes(case):
    from paper_2609_02897_gb300 import asd
    B, n, ctx, page, D = CASES[case]
    Hq, Hkv, cap = 32, 8, 32768
    d = _inputs(B, n, ctx, page, Hq, Hkv, D, cap, case)
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, page, cap,
                         B * cap // page if page else 0, n, n)
    out = _call(d, dims, asd.alloc_workspace(dims, B * n))
    ref = _exact(d, B, n, ctx, page, Hq, Hkv, D)
    assert float((out.double() - ref).norm() / ref.norm()) < BOUND


def test_an_infinite_value_stays_infinite():
    """Both terms of a weight, where it has two, are positive where the weight is: an infinite V
    that every row sees makes its column infinite, and no other."""
    import torch
    from paper_2609_02897_gb300 import asd
    B, n, Hq, Hkv, D, cap = 1, 8, 32, 8, 128, 1024
    d = _inputs(B, n, [700], 0, Hq, Hkv, D, cap, 2)
    d["v_cache"][:, :, 300, 5] = float("inf")
    d["v_cache"][:, :, 2, 77] = -float("inf")
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, 0, cap, 0, n, n)
    out = _call(d, dims, asd.alloc_workspace(dims, n)).float()
    assert bool((out[..., 5] == float("inf")).all()) and bool((out[..., 77] == -float("inf")).all())
    keep = [c for c in range(D) if c not in (5, 77)]
    assert bool(torch.isfinite(out[..., keep]).all())


def test_long_context_step():
    """A step of up to 128 nodes whose attention runs behind the LM head."""
    import torch
    from paper_2609_02897_gb300 import asd
    B, n, Hq, Hkv, D, cap, hidden, vocab = 1, 16, 32, 8, 128, 24576, 64, 200
    ctx = [20000]
    d = _inputs(B, n, ctx, 0, Hq, Hkv, D, cap, 4)
    g = torch.Generator(device="cuda").manual_seed(9)
    d["hidden"] = torch.randn(n, hidden, generator=g, device="cuda").to(torch.bfloat16)
    d["w_lm"] = torch.randn(vocab, hidden, generator=g, device="cuda").to(torch.bfloat16)
    d["tokens"] = torch.randint(0, vocab, (n,), generator=g, device="cuda").int()
    dims = asd.make_dims(B, Hq, Hkv, D, hidden, vocab, asd.ASD_BF16, 0, cap, 0, n, 8)
    out = asd.VerifyStep(dims, n).bind(tau=0.5, **d).run()["attn_out"]
    ref = _exact(d, B, n, ctx, 0, Hq, Hkv, D)
    assert float((out.double() - ref).norm() / ref.norm()) < BOUND
