"""The wide LM head's sharing of node tiles between the CTAs of a cluster, where
it can go wrong: every remainder of four tiles after none, one and two full
rounds, odd and even numbers of 128-row vocabulary tiles per range (a 256-row
tile then straddles two ranges), and hidden widths of one, three and four
64-element k-blocks (up to as many as the ring of three has stages the
accumulators do not alternate, from four on they do).
Bit-compared with the same rows computed by other tile counts: a row's
statistics do not depend on the tile that holds it."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden", [64, 136, 256])
@pytest.mark.parametrize("vocab", [4864, 40000, 45000])
def test_rows_do_not_depend_on_their_tile(hidden, vocab):
    import torch
    from paper_2609_02897_gb300 import asd
    g = torch.Generator(device="cuda").manual_seed(vocab + hidden)
    n = 8
    most = 11 * 128
    h = torch.randn(most, hidden, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(vocab, hidden, generator=g, device="cuda") * 0.1).to(torch.bfloat16)
    tokens = torch.randint(0, vocab, (most,), generator=g, device="cuda").int()
    parent = (torch.arange(most, dtype=torch.int32) % n - 1).cuda()     # chains of 8

    ranges = min(torch.cuda.get_device_properties(0).multi_processor_count, 256, (vocab + 31) // 32)
    clustered = torch.cuda.device_count() == 1 and ranges % 2 == 0

    def call(T):
        dims = asd.make_dims(T // n, 4, 4, 64, hidden, vocab, asd.ASD_BF16, 0, 64, 0, n, n)
        out = {k: torch.zeros(T, dtype=torch.float32, device="cuda")
               for k in ("row_max", "row_lse", "l_draft", "ratio")}
        out["row_argmax"] = torch.zeros(T, dtype=torch.int32, device="cuda")
        out["accept"] = torch.zeros(T, dtype=torch.uint8, device="cuda")
        tiles = -(-T // 128)
        assert asd.asd_lm_head_variant(dims, T, w) == \
            (3 if clustered and (tiles in (3, 4) or tiles >= 7) else 2), tiles
        ws = asd.alloc_workspace(dims, T)
        cu = torch.arange(0, T + 1, n, dtype=torch.int32, device="cuda")
        asd.asd_lmhead_margin(dims, h[:T], w, tokens[:T], parent[:T], cu, 0.5, workspace=ws, **out)
        assert asd.asd_get_device_status(ws) == 0
        return out

    ref = h.float() @ w.float().T
    full = call(most)
    # fp32 sums of bf16 products in another order: 2^-20 of the largest partial sums
    assert float((full["row_max"] - ref.max(1).values).abs().max()) < 1e-4
    assert torch.equal(full["row_argmax"].long(), ref.argmax(1))
    for tiles in (2, 3, 4, 5, 6, 7, 8, 9, 10):
        T = tiles * 128 - (64 if tiles % 2 else 0)
        part = call(T)
        for k, v in part.items():
            assert torch.equal(v.view(torch.uint8), full[k][:T].contiguous().view(torch.uint8)), (tiles, k)
