"""Float MLP stacks that keep their operands in three bf16 planes, at the edges of the product's tiles (256 rows, 32 to 192 columns,
32 of the contraction, planes padded to 64 columns), with pointers that are not 16-byte aligned, and with values at the ends of
the float range, against the oracle or the CUDA-core kernels."""
import os

import pytest
import torch

from oracle import run as orun
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs
from test_gpu_parity import compare, run_gpu

pytestmark = pytest.mark.gpu


def _workload(block, L, d, h, tokens, seed):
    return Workload("t", block, "f32", L=L, d=d, hidden=h, tokens=tokens, batch=1, seq=1, seed=seed, init="small" if block == "postln_mlp" else "")


@pytest.mark.parametrize("block,L,d,h,tokens", [
    ("mlp", 2, 64, 64, 33), ("preln_mlp", 3, 68, 196, 255), ("relu_mlp", 2, 196, 388, 257), ("postln_mlp", 2, 260, 64, 513),
    ("preln_mlp", 2, 64, 1604, 96), ("mlp", 1, 580, 100, 1025), ("preln_mlp", 20, 128, 192, 300),
])
def test_tile_edges_match_oracle(block, L, d, h, tokens):
    w = _workload(block, L, d, h, tokens, 9000 + d + tokens)
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (1, 2))
    assert gpu["ctx"].forms["gemm_parts"] == gpu["ctx"].forms["gemm_f32"] > 0
    compare(w, gpu, orun.run(w, inp, ks=(1, 2), grads_for=("exact", 2)), (1, 2), ("exact", 2))


def _shifted(t):
    """The same values four bytes past a 16-byte boundary."""
    buf = torch.empty(t.numel() + 4, device=t.device, dtype=t.dtype)
    out = buf[1:1 + t.numel()].view(t.shape)
    out.copy_(t)
    return out


def test_weights_and_gradients_at_any_address():
    w = _workload("preln_mlp", 2, 100, 260, 300, 9100)
    inp = make_inputs(w, "cuda")
    got = []
    for shift in (False, True):
        ctx = harness.make_context(w)
        params = {n: _shifted(t) if shift else t for n, t in harness.params_for(w, inp).items()}
        x_all = ctx.forward(params, inp["x0"])
        delta = harness.loss_delta(w, x_all, inp)
        grads = {n: _shifted(t) if shift else t for n, t in ctx.new_grads(with_gate=True).items()}
        g = ctx.backward(params, 1, delta, x_all, grads=grads)
        ctx.sync_status()
        got.append([x_all.clone(), g.clone()] + [grads[n].clone() for n in sorted(grads)])
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("value", [3.4e38, -3.3961e38, float("inf"), float("-inf"), float("nan"), 1e-40])
def test_ends_of_the_float_range(value):
    """A large finite value must not reach the product as an infinite part, an infinity or NaN only where the CUDA cores let it, and
    a value below the parts' range must lose no more than they do.  The value reaches every output of its row through a weight of
    its sign (column 7); what passes by the block, in that column alone, is not compared."""
    w = _workload("mlp", 1, 128, 192, 130, 9200)
    inp = make_inputs(w, "cuda")
    inp["W1"].abs_()
    tiny = abs(value) < 1e-30
    if tiny:
        inp["x0"][5] = value
        inp["W2"].abs_()
    else:
        inp["x0"][5, 7] = value
        inp["W1"][0, :, 7] = -1e-3 if value < 0 else 1e-3
    states = []
    for simt in (False, True):
        if simt:
            os.environ["HBP_FORCE_SIMT"] = "1"
        try:
            ctx = harness.make_context(w)
        finally:
            os.environ.pop("HBP_FORCE_SIMT", None)
        states.append(ctx.forward(harness.params_for(w, inp), inp["x0"])[1].clone())
        ctx.sync_status()
        assert ctx.forms["gemm_simt" if simt else "gemm_parts"] == 2
    got, want = states
    assert torch.equal(torch.isfinite(got), torch.isfinite(want)) and torch.equal(torch.isnan(got), torch.isnan(want))
    got, want = (torch.cat([s[:, :7], s[:, 8:]], 1).double() for s in states)
    # row by row: float sums of the same 128 and 192 terms in another order, 14 roundings of 2^-24 on a random walk of 192
    rows = [r for r in range(w.tokens) if r != 5 or (abs(value) < 1e39 and not tiny)]
    assert torch.isfinite(want[rows]).all()
    assert float(((got[rows] - want[rows]).norm(dim=1) / want[rows].norm(dim=1)).max()) < 14 * 2.0 ** -24
    if abs(value) < 1e39 and not tiny:
        assert float(want[5].norm()) > 1e34  # the value is in every output of its row
    if tiny:
        # parts are multiples of 2^-133, so that the state is off by what is left of it and an activation by up to 2^-134 more
        # (gelu' = 0.5 here); and sums of denormals by up to 2^-150 a term
        left = abs(value - round(value * 2.0 ** 133) * 2.0 ** -133)
        w1, w2 = inp["W1"][0].double(), inp["W2"][0].double()
        off = w2 @ (0.5 * w1.sum(1) * left + 2.0 ** -134) + 320 * 2.0 ** -149
        off = torch.cat([off[:7], off[8:]])
        assert float(off.norm()) < 0.25 * float(want[5].norm())
        assert bool(((got[5] - want[5]).abs() <= off + 14 * 2.0 ** -24 * want[5].abs()).all())
