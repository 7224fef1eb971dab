"""All-step products of the float recurrent kinds that form their left operand while they load it: widths around the edges of
tiles and k-blocks, rows around those of a CTA pair and of a drain, inputs of one to two tiles, unaligned inputs, values at the ends
of the float range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _workload(block, units, in_dim, T, B, loss="every_mse", seed=9500):
    from paper_2501_17086_b200.workloads import Workload
    return Workload("t", block, "f32", L=T, d=2 * units if block == "lstm" else units, hidden=units if block == "lstm" else 0, in_dim=in_dim,
                    batch=B, tokens=B, seed=seed + units + T, loss=loss)


# rows of the products: 1, one short of, exactly and one past a pair's 256; 32 k-blocks (one drain of the gradients) and more
@pytest.mark.parametrize("units,in_dim,T,B,loss", [(32, 4, 1, 1, "every_mse"), (36, 8, 5, 51, "final_mse"), (64, 4, 64, 4, "every_mse"),
                                                   (100, 36, 257, 1, "every_mse"), (128, 260, 41, 25, "every_mse"),
                                                   (260, 32, 16, 129, "final_mse"), (516, 20, 6, 43, "every_mse")])
@pytest.mark.parametrize("block", ["rnn_tanh", "gru", "lstm"])
def test_cell_products_match_the_oracle(block, units, in_dim, T, B, loss):
    from oracle import run as orun
    from paper_2501_17086_b200.workloads import make_inputs
    from test_gpu_parity import compare, run_gpu
    w = _workload(block, units, in_dim, T, B, loss)
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (2,))
    assert gpu["ctx"].forms["gemm_cell"] == min(2, T) + 2   # the VJPs, the gradients of the truncated and of the exact pass
    compare(w, gpu, orun.run(w, inp, ks=(2,), grads_for=("exact", 2)), (2,), ("exact", 2))


def _grads(w, inp, scale=1.0, xin=None, poke=None):
    """Parameter gradients and iterate of backward(1) from a loss gradient times `scale`; `poke` changes that gradient."""
    from paper_2501_17086_b200 import harness
    ctx = harness.make_context(w)
    params = harness.params_for(w, inp)
    xin = harness.rnn_inputs(w, inp) if xin is None else xin
    x = ctx.forward(params, inp["x0"], xin)
    delta = harness.loss_delta(w, x, inp) * scale
    if poke is not None:
        poke(delta)
    grads = ctx.new_grads(with_gate=True)
    g = ctx.backward(params, 1, delta, x, xin, grads=grads)
    ctx.sync_status()
    assert ctx.forms["gemm_cell"] == 2
    return g.clone(), {n: t.clone() for n, t in grads.items()}


@pytest.mark.parametrize("block", ["rnn_tanh", "gru", "lstm"])
def test_cell_products_take_inputs_of_any_alignment(block):
    from paper_2501_17086_b200 import harness
    from paper_2501_17086_b200.workloads import make_inputs
    w = _workload(block, 48, 12, 30, 11)
    inp = make_inputs(w, "cuda")
    X = harness.rnn_inputs(w, inp)
    shifted = torch.empty(X.numel() + 1, device="cuda")[1:].view_as(X).copy_(X)
    a, b = _grads(w, inp), _grads(w, inp, xin=shifted)
    assert torch.equal(a[0], b[0])
    for n in a[1]:
        assert torch.equal(a[1][n], b[1][n]), n


@pytest.mark.parametrize("block", ["rnn_tanh", "gru", "lstm"])
@pytest.mark.parametrize("power", [-100, -60, 100, 118])
def test_cell_products_hold_at_the_ends_of_the_float_range(block, power):
    """The backward pass is linear in the loss gradient: scaled by a power of two, its results scale by the same, whether the parts of
    the operand would run into the denormals (2^-100 leaves the least of them above 2^-126) or overflow (2^103 and more)."""
    from paper_2501_17086_b200.workloads import make_inputs
    w = _workload(block, 48, 12, 30, 11)
    inp = make_inputs(w, "cuda")
    a, b = _grads(w, inp), _grads(w, inp, scale=2.0 ** power)
    for x, y in [(a[0], b[0])] + [(a[1][n], b[1][n]) for n in a[1]]:
        x, y = x.double(), y.double() * 2.0 ** -power
        # float sums in another order where a sum is formed again: a relative rounding of each of some 330 additions, at random
        assert float((x - y).norm() / x.norm()) < 2e-6


@pytest.mark.parametrize("block", ["rnn_tanh", "gru", "lstm"])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_cell_products_carry_what_is_not_finite(block, value):
    """One infinite (or NaN) element of the loss gradient of the last state: rows of other sequences keep their bits, and the row's
    own and the weight gradients are not finite where plain float arithmetic says so."""
    from paper_2501_17086_b200.workloads import make_inputs
    w = _workload(block, 48, 12, 30, 11)
    inp = make_inputs(w, "cuda")

    def poke(delta):
        delta[-1, 3, 5] = value

    (g0, d0), (g1, d1) = _grads(w, inp), _grads(w, inp, poke=poke)
    others = [b for b in range(11) if b != 3]
    assert torch.equal(g0[:, others], g1[:, others])
    assert not torch.isfinite(g1[-2, 3]).all()
    assert not torch.isfinite(d1["dW"]).all() and not torch.isfinite(d1["dU"]).all()
    rows = torch.isfinite(d1["dU"]).all(dim=1)   # operand channels that the element does not reach
    assert torch.allclose(d0["dU"][rows], d1["dU"][rows], rtol=1e-5, atol=1e-6 * float(d0["dU"].abs().max()))


def _step(block, x, xt, W, U, a):
    """One step's next state, in 64 bits (`xt` the inputs of the same rows)."""
    if block == "rnn_tanh":
        return a * x + torch.tanh(x @ W.T + xt @ U.T)
    if block == "gru":
        (ur, uz, un), (wr, wz, wn) = (xt @ U.T).chunk(3, -1), (x @ W.T).chunk(3, -1)
        z = torch.sigmoid(uz + wz)
        return z * x + (1 - z) * torch.tanh(un + torch.sigmoid(ur + wr) * wn)
    c, h = x.chunk(2, -1)
    i, f, g, o = (xt @ U.T + h @ W.T).chunk(4, -1)
    c = torch.sigmoid(f) * c + torch.sigmoid(i) * torch.tanh(g)
    return torch.cat([c, torch.sigmoid(o) * torch.tanh(c)], -1)


# Rows of the product a multiple of 4: 32 additions a chain in the tensor core, each of which loses up to 2^-23 of a partial sum, that is on
# average half as large as the whole: 32 * 2^-23 / 4.  Else sums of floats: 16 rounded additions a set, at random, 4 * 2^-24.  The tanh RNN's
# coefficients 1 - tanh^2 were formed from states not yet rounded to floats, which here they are: 2 |tanh| |W row| |x| 2^-25, 4 * 2^-24 at most.
@pytest.mark.parametrize("T,B", [(500, 132), (499, 131), (499, 130), (33, 3), (17, 1), (5, 3)])
# states and inputs in one tile together, in two, in one and more each, the last of them with columns past their end
@pytest.mark.parametrize("units,in_dim", [(64, 12), (96, 100), (164, 128), (256, 8), (300, 40), (452, 180)])
@pytest.mark.parametrize("block", ["rnn_tanh", "gru", "lstm"])
def test_weight_gradients_are_as_exact_as_their_rows_allow(block, units, in_dim, T, B):
    """Against 64 bits from the pass's own states and iterate, so that little but the products' sums is compared."""
    from paper_2501_17086_b200 import harness
    from paper_2501_17086_b200.workloads import make_inputs
    w = _workload(block, units, in_dim, T, B)
    inp = make_inputs(w, "cuda")
    ctx, params, X = harness.make_context(w), harness.params_for(w, inp), harness.rnn_inputs(w, inp)
    x = ctx.forward(params, inp["x0"], X)
    delta = harness.loss_delta(w, x, inp)
    grads = ctx.new_grads()
    g = ctx.backward(params, 1, delta, x, X, grads=grads)
    ctx.sync_status()
    assert ctx.forms["gemm_cell"] == 2
    W, U = (params[n].double().requires_grad_() for n in ("W", "U"))
    rows = lambda t: t.reshape(T * B, -1).double()
    out = _step(block, rows(x[:-1]), rows(X), W, U, params["a"].double() if "a" in params else None)
    for name, ref in zip(("dW", "dU"), torch.autograd.grad(out, (W, U), rows(g[1:]))):
        bound = (32 * 2.0 ** -23 / 4 if T * B % 4 == 0 else 4 * 2.0 ** -24) + (4 * 2.0 ** -24 if block == "rnn_tanh" else 0)
        assert float((grads[name] - ref).norm() / ref.norm()) < bound, name


@pytest.mark.parametrize("block,units,in_dim", [("gru", 64, 64), ("lstm", 64, 64), ("rnn_tanh", 512, 512)])
def test_weight_gradients_of_more_rows_than_sets_have_room(block, units, in_dim):
    """Up to 57 rounded additions a set instead of 16.  Each is off by 2^-25 / sqrt(3) of a partial sum at the root mean square, which grows as
    the root of their number: 57 of them sqrt(57 / 2) 2^-25 / sqrt(3) = 1.5 * 2^-24, so that the same bound holds."""
    test_weight_gradients_are_as_exact_as_their_rows_allow(block, units, in_dim, 1023, 129)
