"""The one-launch recurrences (forward pass and exact backpropagation of the recurrent cells) at the edges of their
splits: one row, a ninth row beside a tile of eight, two and three tiles of rows, units that leave padding in the last
8-unit tile or the last CTA, weights that do not fit shared memory, one and two steps."""
import os

import pytest
import torch

from oracle import run as orun
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs
from test_gpu_parity import compare, run_gpu

pytestmark = pytest.mark.gpu


def _workload(block, dtype, T, u, B, nin, loss="every_mse"):
    return Workload("t", block, dtype, L=T, d=2 * u if block == "lstm" else u, hidden=u if block == "lstm" else 0, in_dim=nin,
                    batch=B, tokens=B, seed=7000 + T + u + B, loss=loss)


def _forward(w, inp, form):
    """The states, from a context whose forward pass has to take ``form`` (one launch, or one per step)."""
    ctx = harness.make_context(w)
    x = ctx.forward(harness.params_for(w, inp), inp["x0"], harness.rnn_inputs(w, inp))
    ctx.sync_status()
    assert _recurrences(ctx) == {form: w.L if form == "step" else 1}
    return x


def _recurrences(ctx):
    return {n: c for n, c in ctx.forms.items() if c and n in ("cell_cluster", "rnn_cluster", "rnn_four_rows", "step")}


@pytest.mark.parametrize("block,dtype,T,u,B,nin", [
    ("gru", "f32", 1, 4, 1, 4), ("gru", "f32", 2, 8, 9, 4), ("gru", "f32", 5, 100, 37, 20), ("gru", "f32", 6, 132, 192, 64),
    ("gru", "f32", 3, 512, 130, 212), ("gru", "f32", 3, 512, 200, 36), ("gru", "bf16", 4, 72, 19, 16),
    ("lstm", "f32", 1, 4, 1, 4), ("lstm", "f32", 2, 12, 9, 8), ("lstm", "f32", 5, 200, 100, 32), ("lstm", "f32", 3, 512, 128, 212),
    ("lstm", "f32", 3, 372, 150, 100), ("lstm", "bf16", 4, 40, 26, 8),
    ("rnn_tanh", "f32", 1, 4, 1, 4), ("rnn_tanh", "f32", 6, 68, 50, 12), ("rnn_tanh", "f32", 4, 508, 180, 256),
    ("rnn_tanh", "f32", 4, 512, 190, 8), ("rnn_tanh", "bf16", 5, 264, 17, 40),
    # more units: 72 to 96 per CTA, all weights streamed, blocks of padding in the backward contraction
    ("gru", "f32", 2, 1100, 10, 20), ("gru", "f32", 2, 1536, 9, 16), ("lstm", "f32", 2, 1300, 60, 8), ("lstm", "f32", 2, 1536, 8, 4),
])
def test_edges_of_the_splits_match_oracle(block, dtype, T, u, B, nin):
    w = _workload(block, dtype, T, u, B, nin)
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (1,))
    # one forward and one exact pass, each one launch
    assert _recurrences(gpu["ctx"]) == ({"rnn_cluster": 1, "cell_cluster": 1} if block == "rnn_tanh" else {"cell_cluster": 2})
    compare(w, gpu, orun.run(w, inp, ks=(1,), grads_for=("exact", 1)), (1,), ("exact", 1))


@pytest.mark.parametrize("dtype,T,u,B,nin", [
    ("f32", 300, 512, 32, 256), ("f32", 100, 512, 190, 8), ("f32", 200, 256, 40, 64), ("f32", 120, 128, 201, 20), ("bf16", 60, 256, 33, 16),
    ("f32", 200, 100, 50, 20), ("f32", 100, 508, 180, 256), ("f32", 50, 4, 5, 4), ("f32", 64, 436, 100, 36), ("bf16", 80, 264, 17, 40),
])
def test_tanh_rnn_forms_agree_bit_for_bit(dtype, T, u, B, nin):
    """The forward recurrence amplifies rounding, so its forms keep one order of sums per width: many rows at once against
    four at a time (128, 256 and 512 units), or against one launch per step."""
    w = _workload("rnn_tanh", dtype, T, u, B, nin)
    inp = make_inputs(w, "cuda")
    x = _forward(w, inp, "rnn_cluster")
    if u in (128, 256, 512):
        for r in range(0, B, 4):
            n = min(4, B - r)
            part = dict(inp, X=inp["X"][:, r:r + n].contiguous(), x0=inp["x0"][r:r + n].contiguous())
            assert torch.equal(_forward(_workload("rnn_tanh", dtype, T, u, n, nin), part, "rnn_four_rows"), x[:, r:r + n])
    else:
        os.environ["HBP_FORCE_SIMT"] = "1"
        try:
            assert torch.equal(_forward(w, inp, "step"), x)
        finally:
            del os.environ["HBP_FORCE_SIMT"]


@pytest.mark.parametrize("block", ["gru", "lstm"])
def test_unaligned_weights_take_the_per_step_form(block):
    """Weights that start 4 bytes past a 16-byte boundary: the one-launch forms read them in vectors and decline."""
    w = _workload(block, "f32", 9, 20, 11, 8)
    inp = make_inputs(w, "cuda")
    moved = torch.empty(inp["W"].numel() + 1, device="cuda")[1:].view_as(inp["W"])
    moved.copy_(inp["W"])
    x, y = _forward(w, inp, "cell_cluster"), _forward(w, dict(inp, W=moved), "step")
    assert float((x - y).norm() / x.norm()) < 1e-6


def test_exact_pass_of_wide_tanh_rnns_is_one_launch():
    w = _workload("rnn_tanh", "f32", 2, 1536, 40, 8)
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (1,))
    assert gpu["ctx"].forms["cell_cluster"] == 1   # (the forward pass of that width is step by step)
    compare(w, gpu, orun.run(w, inp, ks=(1,), grads_for=("exact", 1)), (1,), ("exact", 1))


@pytest.mark.parametrize("u", [12, 100])
def test_an_infinite_gradient_stays_infinite_beside_padding_units(u):
    """Exact backpropagation of a tanh RNN with weights >= 0 (tanh' > 0): an infinite gradient of one unit makes all gradients of
    its row infinite from the step before on, and no NaN, also where the last 8-unit tile has padding."""
    w = _workload("rnn_tanh", "f32", 6, u, 9, 8)
    inp = make_inputs(w, "cuda")
    inp["W"].abs_().mul_(0.1)
    params, xin = harness.params_for(w, inp), harness.rnn_inputs(w, inp)
    ctx = harness.make_context(w)
    x = ctx.forward(params, inp["x0"], xin)
    delta = torch.ones_like(x)
    delta[-1, 4, 2] = float("inf")
    g = ctx.exact(params, delta, x, xin)
    ctx.sync_status()
    assert ctx.forms["cell_cluster"] == 1 and ctx.forms["step"] == 0
    assert torch.isposinf(g[:-1, 4]).all()
    others = [r for r in range(9) if r != 4]
    assert torch.isfinite(g[:, others]).all()
