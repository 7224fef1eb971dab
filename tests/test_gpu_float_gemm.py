"""The float tensor-core GEMMs at the edges of their tiles: rows, columns and contraction lengths around 32 and 128, every
orientation of the operands and every epilogue of the float MLP and decoder kinds, against the oracle.  Each test runs on the kernel
that splits its operands into three bf16 parts itself, and on the one that reads them already split where a stack keeps them so."""
import os

import pytest
import torch

from oracle import run as orun
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs
from test_gpu_parity import compare, rel_l2, run_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(params=["split_inside", "planes"], autouse=True)
def operands(request, monkeypatch):
    """HBP_GEMM_PAIR=0 contexts split inside the kernel.  Every context that a test made has to have taken the products meant."""
    made, make = [], harness.make_context

    def make_context(w):
        made.append((w, make(w), os.environ.get("HBP_FORCE_SIMT") == "1"))
        return made[-1][1]

    monkeypatch.setattr(harness, "make_context", make_context)
    if request.param == "split_inside":
        monkeypatch.setenv("HBP_GEMM_PAIR", "0")
    yield request.param
    for w, ctx, simt in made:
        kept = request.param == "planes" and not simt and w.tokens > 32 and w.d >= 64 and w.hidden >= 64
        assert ctx.forms["gemm_parts"] == (ctx.forms["gemm_f32"] if kept else 0)
        assert not simt or ctx.forms["gemm_f32"] == 0


@pytest.mark.parametrize("block,L,d,h,tokens", [
    ("mlp", 2, 4, 8, 33), ("mlp", 2, 128, 256, 127), ("mlp", 3, 132, 260, 129), ("preln_mlp", 2, 36, 388, 257),
    ("preln_mlp", 2, 260, 124, 1000), ("relu_mlp", 2, 100, 132, 70), ("postln_mlp", 2, 132, 300, 161), ("mlp", 1, 1028, 1032, 40),
    ("relu_mlp", 2, 388, 36, 257), ("postln_mlp", 2, 60, 520, 130),
])
def test_tile_edges_match_oracle(block, L, d, h, tokens):
    w = Workload("t", block, "f32", L=L, d=d, hidden=h, tokens=tokens, batch=1, seq=1, seed=8000 + d + tokens)
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (1, L))
    # forward: two products a layer; each pass: two per VJP over all layers (k of them, the exact pass one per layer) and, for the
    # parameters, one VJP's first product again (not in the exact pass) and two batched weight gradients
    forward = [(tokens, h, d), (tokens, d, h)] * L
    vjp, weights = [(tokens, h, d), (tokens, d, h)], [(d, h, tokens), (h, d, tokens)]
    products = forward + vjp * (1 + L) + ([vjp[0]] + weights) * 2 + vjp * L + weights
    taken = sum(m > 32 and k > 16 for m, n, k in products)
    assert gpu["ctx"].forms["gemm_f32"] == taken and gpu["ctx"].forms["gemm_simt"] == len(products) - taken
    compare(w, gpu, orun.run(w, inp, ks=(1, L), grads_for=("exact", L)), (1, L), ("exact", L))


@pytest.mark.parametrize("L,d,h,tokens", [
    (2, 64, 256, 12), (2, 64, 256, 32), (2, 132, 260, 16), (2, 32, 128, 400), (2, 12, 64, 300), (2, 24, 520, 200), (2, 64, 96, 40),
    (2, 256, 520, 100), (2, 520, 1560, 300), (8, 64, 128, 200), (8, 72, 200, 64), (8, 128, 256, 200), (8, 180, 500, 1000),
])
def test_no_further_from_64_bits_than_float_sums(L, d, h, tokens):
    """Splitting the operands must not cost precision, neither in short contractions nor by a bias that adds up over the layers:
    states, gradients and weight gradients of a float MLP are no further from the oracle than on the CUDA cores (10 % for
    chance: norms over at least a thousand elements)."""
    w = Workload("t", "mlp", "f32", L=L, d=d, hidden=h, tokens=tokens, batch=1, seq=1, seed=8400 + d + tokens)
    inp = make_inputs(w, "cuda")
    ref = orun.run(w, inp, ks=(1,), grads_for=("exact",))
    off = []
    for simt in (False, True):
        if simt:
            os.environ["HBP_FORCE_SIMT"] = "1"
        try:
            gpu = run_gpu(w, inp, (1,))
        finally:
            os.environ.pop("HBP_FORCE_SIMT", None)
        got = {"x": (gpu["x"][-1], ref["xs"][-1]), "g": (gpu["exact"][0], ref["exact"][0])}
        got.update({n: (gpu["grads"]["exact"]["d" + n], v) for n, v in ref["grads"]["exact"].items()})
        off.append({n: rel_l2(to_np(a), b) for n, (a, b) in got.items()})
    for n in off[0]:
        assert off[0][n] <= 1.1 * off[1][n], (n, off)


def test_non_finite_inputs_stay_non_finite():
    """An infinity and a NaN reach the same rows as in the CUDA-core kernel, a value next to the largest float none."""
    w = Workload("t", "mlp", "f32", L=1, d=64, hidden=160, tokens=200, batch=1, seq=1, seed=8100)
    inp = make_inputs(w, "cuda")
    inp["x0"][3, 5], inp["x0"][77, 0], inp["x0"][150, 63] = float("inf"), float("nan"), -3.4e38
    finite = []
    for simt in (False, True):
        if simt:
            os.environ["HBP_FORCE_SIMT"] = "1"
        try:
            ctx = harness.make_context(w)
        finally:
            os.environ.pop("HBP_FORCE_SIMT", None)
        finite.append(torch.isfinite(ctx.forward(harness.params_for(w, inp), inp["x0"])))
        ctx.sync_status()
        assert ctx.forms["gemm_simt" if simt else "gemm_f32"] == 2
    assert torch.equal(finite[0][0], finite[1][0])
    assert torch.equal(finite[0][1].all(dim=1), finite[1][1].all(dim=1))


def test_infinities_and_nans_have_the_value_a_plain_sum_gives():
    """Weights of one sign per row, so that an infinite state element makes whole rows of the next state +inf or -inf (in three
    products of parts an infinity meets remainders that are zero or of the other sign: NaN); 0.5 is exact in the tensor core's
    type, the NaN's payload lies only in the bits it drops, and -3.4e38 is next to the largest float."""
    w = Workload("t", "mlp", "f32", L=1, d=256, hidden=320, tokens=200, batch=1, seq=1, seed=8200)
    inp = make_inputs(w, "cuda")
    sign = torch.where(torch.arange(w.d, device="cuda") % 3 == 0, -1.0, 1.0)
    inp["W1"].abs_()
    inp["W1"][0, :160] = 0.5
    inp["W2"].abs_().mul_(sign[None, :, None])
    x0 = inp["x0"].abs_()
    x0[3, 5], x0[40, 1], x0[150, 63] = float("inf"), float("inf"), -3.4e38
    x0.view(torch.int32)[77, 0] = 0x7f800001
    states = []
    for simt in (False, True):
        if simt:
            os.environ["HBP_FORCE_SIMT"] = "1"
        try:
            ctx = harness.make_context(w)
        finally:
            os.environ.pop("HBP_FORCE_SIMT", None)
        states.append(ctx.forward(harness.params_for(w, inp), x0)[1].clone())
        ctx.sync_status()
        assert ctx.forms["gemm_simt" if simt else "gemm_f32"] == 2
    got, want = states
    assert torch.isinf(want[3]).all() and torch.isinf(want[40]).all() and torch.isnan(want[77]).all()
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.isinf(got), torch.isinf(want))
    assert torch.equal(got[torch.isinf(want)], want[torch.isinf(want)])   # the signs
    rest = torch.isfinite(want)
    rest[150] = False
    assert float((got[rest] - want[rest]).norm() / want[rest].norm()) < 1e-6
