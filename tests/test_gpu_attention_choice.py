"""Which bf16 kernel a call of up to 128 nodes runs, told by its bits: what the
mma.sync kernel writes depends neither on the cache's capacity nor on whether an
LM head runs beside it, and the tensor-core kernel rounds otherwise."""
import math

import pytest

from test_gpu_attention_precision import BOUND, _exact
from test_gpu_attention_ragged import _call, _inputs

pytestmark = pytest.mark.gpu


def _same(a, b):
    import torch
    return torch.equal(a.view(torch.int16), b.view(torch.int16))


def _tight(d, cap, page):
    """The same contexts in a cache of `cap` slots per sequence."""
    if page:
        return dict(d, page_table=d["page_table"][:, :cap // page].contiguous())
    return dict(d, **{k: d[k][:, :, :cap].contiguous() for k in ("k_cache", "v_cache")})


def _alone(d, B, n, page, pages, cap, Hq, Hkv, D):
    from paper_2609_02897_gb300 import asd
    dims = asd.make_dims(B, Hq, Hkv, D, 64, 64, asd.ASD_BF16, page, cap, pages, n, n)
    return _call(d, dims, asd.alloc_workspace(dims, B * n))


def _beside_lm_head(d, B, n, page, pages, cap, Hq, Hkv, D, hidden=4096, vocab=128000):
    """attn_out of a step; its LM head (by default 1 GB of weight) hides attention
    of up to 0.8 key tiles a microsecond (contiguous, D = 128)."""
    import torch
    from paper_2609_02897_gb300 import asd
    dims = asd.make_dims(B, Hq, Hkv, D, hidden, vocab, asd.ASD_BF16, page, cap, pages, n, n)
    bf16 = dict(dtype=torch.bfloat16, device="cuda")
    step = asd.VerifyStep(dims, B * n).bind(
        tau=0.5, hidden=torch.zeros(B * n, hidden, **bf16), w_lm=torch.zeros(vocab, hidden, **bf16),
        tokens=torch.zeros(B * n, dtype=torch.int32, device="cuda"), **d)
    return step.run()["attn_out"]


def _waves(B, Hkv):
    import torch
    return math.ceil(B * Hkv / torch.cuda.get_device_properties(0).multi_processor_count)


def _limit(k, page, D, both):
    """Key tiles of 32 up to which the mma.sync kernel takes a call of k items per SM."""
    by_cache = (1.0 if page == 0 else 0.8 if page >= 32 else 0.65) * (2.0 if D == 64 else 1.0)
    return int(by_cache * ((17.0 if both else 23.0) * k - 18.0) / (k + 1.6))


SHAPES = [(128, 1, 0, 32, 128), (64, 2, 16, 32, 128), (60, 2, 0, 32, 64), (96, 1, 64, 24, 128)]


@pytest.mark.parametrize("B,n,page,Hq,D", SHAPES + [(20, 6, 0, 32, 64)])
def test_many_short_sequences_in_a_tight_cache(B, n, page, Hq, D):
    Hkv, cap = 8, 64
    ctx = [1 + (b * 37) % 40 for b in range(B)]
    d = _inputs(B, n, ctx, page, Hq, Hkv, D, cap, B)
    pages = B * cap // page if page else 0
    out = _alone(d, B, n, page, pages, cap, Hq, Hkv, D)
    # the step commits to the cache, past the contexts
    assert _same(out, _beside_lm_head(d, B, n, page, pages, cap, Hq, Hkv, D))


@pytest.mark.parametrize("B,n,page,Hq,D", SHAPES)
def test_a_large_cache_leaves_it_to_the_contexts(B, n, page, Hq, D):
    """From three items per SM on: equal contexts at the limit's last tile and one
    key beyond; one sequence too long for the mma.sync kernel alone; long ones."""
    Hkv, cap = 8, 2048
    k = _waves(B, Hkv)
    assert k >= 3
    limit = _limit(k, page, D, True)
    last = 32 * (limit - 1)          # the tree's tile makes the limit
    pages = B * cap // page if page else 0
    short = 32 * (_limit(k, page, D, False) - 1) // 64 * 64
    assert last + 1 <= short
    for ctx, mma in (([last] * B, True), ([last + 1] * B, False),
                     ([1] * (B - 1) + [32 * (2 * limit - 1)], True),
                     ([1] * (B - 1) + [32 * (2 * limit - 1) + 1], False)):
        d = _inputs(B, n, ctx, page, Hq, Hkv, D, cap, B)
        out = _alone(d, B, n, page, pages, cap, Hq, Hkv, D)
        if max(ctx) <= short:        # the tight cache takes the mma.sync kernel
            ref = _alone(_tight(d, short, page), B, n, page, pages, short, Hq, Hkv, D)
            assert _same(out, ref) == mma
        else:                        # the short sequences' rows, as in a tight cache
            t = _tight(d, 64, page)
            t["ctx_len"] = d["ctx_len"].clamp(max=1)
            ref = _alone(t, B, n, page, pages, 64, Hq, Hkv, D)
            assert _same(out[:(B - 1) * n], ref[:(B - 1) * n]) == mma
    ctx = [1500 + b for b in range(B)]
    d = _inputs(B, n, ctx, page, Hq, Hkv, D, cap, B)
    out = _alone(d, B, n, page, pages, cap, Hq, Hkv, D)
    exact = _exact(d, B, n, ctx, page, Hq, Hkv, D)
    assert float((out.double() - exact).norm() / exact.norm()) < BOUND   # 2.2e-3: mma.sync


# (B, nodes, hidden, vocab, contexts at the limit, and one key beyond).  A tiny LM
# head: 16 key tiles on the busiest SM, which are the longest split's (84 context
# tiles in 6 splits, 2 of the tree).  One of 480 MB: 60 tiles, those of one
# unsplit sequence among 40 (the others share out 1 tile per SM each).
STEPS = [
    (2, 40, 64, 200, [2688, 2688], [2688, 2689]),
    (40, 3, 4096, 58600, [1] * 39 + [32 * 59], [1] * 39 + [32 * 59 + 1]),
    (2, 40, 64, 200, [0, 5], [4000, 40]),
]


@pytest.mark.parametrize("case", range(len(STEPS)))
def test_a_step_runs_the_kernel_its_contexts_call_for(case):
    """Up to the limit the mma.sync kernel beside the LM head, with the bits of a
    step whose LM head hides any context of the cache; beyond it the tensor-core
    kernel, with those of an attention call by itself."""
    B, n, hidden, vocab, at, beyond = STEPS[case]
    Hq, Hkv, D, cap = 16, 4, 128, 4096 if B == 2 else 2048
    for ctx, mma in ((at, True), (beyond, False)):
        d = _inputs(B, n, ctx, 0, Hq, Hkv, D, cap, case)
        alone = _alone(d, B, n, 0, 0, cap, Hq, Hkv, D)
        out = _beside_lm_head(d, B, n, 0, 0, cap, Hq, Hkv, D, hidden, vocab).clone()
        # the step has committed past the contexts, which no attention reads
        hidden_by_lm = _beside_lm_head(d, B, n, 0, 0, cap, Hq, Hkv, D)
        assert not _same(alone, hidden_by_lm)
        assert _same(out, hidden_by_lm if mma else alone)
