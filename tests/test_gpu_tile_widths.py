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


@pytest.mark.parametrize("block,rows", [("preln_mlp", 65), ("preln_mlp", 130), ("preln_mlp", 1003), ("postln_mlp", 259), ("preln_transformer", 3 * 91)])
def test_weight_gradients_of_any_number_of_rows_run_on_the_tensor_cores(block, rows, monkeypatch):
    """The contraction of a weight gradient runs over the rows: its ragged end, in a block of 64 in part, against the CUDA cores."""
    from paper_2501_17086_b200 import harness
    from paper_2501_17086_b200.workloads import Workload, make_inputs
    tr = block == "preln_transformer"
    w = Workload("t", block, "bf16", L=2, d=128, hidden=264, n_heads=2 if tr else 0, head_dim=64 if tr else 0, seq=91 if tr else 1, batch=3 if tr else 1,
                 tokens=rows, seed=9750 + rows, init="small" if block == "postln_mlp" else "")
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    ctx = harness.make_context(w)
    x = ctx.forward(params, inp["x0"])
    delta = harness.loss_delta(w, x, inp)
    grads = ctx.new_grads()
    g = ctx.backward(params, 1, delta, x, grads=grads)
    ctx.sync_status()
    assert ctx.forms["gemm_simt"] == 0
    # dW2 = G^T gelu(Z), the sums over the rows in 64 bits from the same bf16 estimates; gelu(Z) formed again, so bf16's 2^-9 each
    h0 = x[0].double() if block == "postln_mlp" else torch.nn.functional.layer_norm(x[1 if tr else 0].double(), (128,), eps=w.ln_eps)
    if block != "postln_mlp":
        act = torch.nn.functional.gelu(h0 @ params["W1"][0].double().T)
        ref = g[2 if tr else 1].double().T @ act
        assert float((grads["dW2"][0].double() - ref).norm() / ref.norm()) < 2e-2
    monkeypatch.setenv("HBP_FORCE_SIMT", "1")
    plain = harness.make_context(w)
    plain.forward(params, inp["x0"])
    other = plain.new_grads()
    plain.backward(params, 1, delta, x, grads=other)
    for n in grads:
        assert float((grads[n] - other[n]).norm() / other[n].norm()) < 2e-2, n
