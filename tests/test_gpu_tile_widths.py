"""bf16 products on CTA pairs whose tiles are narrower than 256 columns: every width that the rule may choose, last tiles in part, on
row counts around a pair's 256.  An output is the same sum in the same order whatever the tile, so single CTAs give the same bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block,d,h,tokens,seq", [
    ("preln_mlp", 768, 3072, 1000, 0), ("preln_mlp", 512, 2048, 2664, 0), ("preln_mlp", 264, 520, 257, 0), ("preln_mlp", 1000, 3000, 511, 0),
    ("postln_mlp", 328, 1032, 700, 0), ("preln_mlp", 136, 4096, 513, 0), ("preln_transformer", 512, 2048, 8 * 111, 111),
    ("preln_transformer", 192, 776, 3 * 250, 250)])
def test_narrow_tiles_give_the_bits_of_single_ctas(block, d, h, tokens, seq, monkeypatch):
    from paper_2501_17086_b200 import harness
    from paper_2501_17086_b200.workloads import Workload, make_inputs
    tr = block == "preln_transformer"
    w = Workload("t", block, "bf16", L=2, d=d, hidden=h, n_heads=d // 64 if tr else 0, head_dim=64 if tr else 0, seq=seq if tr else 1,
                 batch=tokens // seq if tr else 1, tokens=tokens, seed=9700 + d, init="small" if block == "postln_mlp" else "")
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    outs = []
    for pair in ("1", "0"):
        monkeypatch.setenv("HBP_GEMM_PAIR", pair)
        ctx = harness.make_context(w)
        x = ctx.forward(params, inp["x0"])
        delta = harness.loss_delta(w, x, inp)
        got = {"x": x.clone()}
        for exact in (False, True):
            grads = ctx.new_grads()
            got[exact] = (ctx.exact(params, delta, x, grads=grads) if exact else ctx.backward(params, 2, delta, x, grads=grads)).clone()
            got.update({(exact, n): t for n, t in grads.items()})
        ctx.sync_status()
        outs.append(got)
    for key, value in outs[0].items():
        assert torch.equal(value, outs[1][key]), key
