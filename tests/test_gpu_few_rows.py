"""Float MLP stacks of few rows as one launch a pass: rows that fill a cluster's three in part, hidden units that leave CTAs without any,
more layers than CTAs, widths at both ends of the rule, every gate and loss."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", ["mlp", "preln_mlp"])
@pytest.mark.parametrize("L,d,h,rows", [(1, 4, 4, 1), (8, 64, 256, 32), (3, 12, 20, 5), (17, 100, 36, 31), (9, 256, 256, 6), (2, 388, 124, 3), (20, 32, 2048, 4)])
def test_few_rows_match_the_oracle(block, L, d, h, rows):
    from oracle import run as orun
    from paper_2501_17086_b200.workloads import Workload, make_inputs
    from test_gpu_parity import compare, run_gpu
    w = Workload("t", block, "f32", L=L, d=d, hidden=h, tokens=rows, batch=1, seq=1, seed=9800 + d, loss="final_mse")
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (0, 1, 3))
    assert gpu["ctx"].forms["few_rows"] == 5   # the forward pass, three backward passes and the exact one
    compare(w, gpu, orun.run(w, inp, ks=(0, 1, 3), grads_for=("exact", 3)), (0, 1, 3), ("exact", 3))


@pytest.mark.parametrize("gate", ["one", "shared", "per_step"])
@pytest.mark.parametrize("every", [False, True])
@pytest.mark.parametrize("block,L,d,h,rows", [("mlp", 5, 36, 100, 7), ("preln_mlp", 19, 64, 96, 30)])
def test_few_rows_agree_with_a_launch_per_product(gate, every, block, L, d, h, rows, monkeypatch):
    from paper_2501_17086_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + rows)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")
    params = {"W1": rand(L, h, d) / d ** 0.5, "W2": rand(L, d, h) * (0.5 / h ** 0.5)}
    if gate != "one":
        params["a"] = 0.7 + 0.3 * torch.rand((d,) if gate == "shared" else (L, d), generator=gen, device="cuda")
    x0, delta = rand(rows, d), rand(L + 1, rows, d) if every else rand(rows, d)
    cfg = B.make_config(block, "f32", L, d, rows, hidden=h, gate={"one": B.GATE_ONE, "shared": B.GATE_CHANNEL_SHARED, "per_step": B.GATE_CHANNEL_PER_STEP}[gate],
                        loss=B.LOSS_EVERY_STEP if every else B.LOSS_FINAL)
    outs = []
    for simt in ("0", "1"):
        monkeypatch.setenv("HBP_FORCE_SIMT", simt)
        ctx = B.Context(cfg)
        got = {"x": ctx.forward(params, x0)}
        for k in (1, 2):
            grads = ctx.new_grads(with_gate=True)
            got[k] = ctx.backward(params, k, delta, got["x"], grads=grads)
            got.update({(k, n): t for n, t in grads.items()})
        grads = ctx.new_grads(with_gate=True)
        got["exact"] = ctx.exact(params, delta, got["x"], grads=grads)
        got.update({("exact", n): t for n, t in grads.items()})
        got["without"] = ctx.backward(params, 2, delta, got["x"])   # no parameter gradients asked for
        got["exact without"] = ctx.exact(params, delta, got["x"])
        ctx.sync_status()
        assert ctx.forms["few_rows"] == (0 if simt == "1" else 6)
        outs.append(got)
    assert torch.equal(outs[0]["without"], outs[0][2]) and torch.equal(outs[0]["exact without"], outs[0]["exact"])
    for key, value in outs[0].items():  # each within some 5e-7 of the sums in 64 bits
        ref = outs[1][key]
        assert float((value - ref).norm() / ref.norm()) < 2e-6, key


@pytest.mark.parametrize("gate", ["one", "shared", "per_step"])
@pytest.mark.parametrize("block", ["mlp", "preln_mlp"])
def test_scans_round_a_state_only_where_it_is_stored(block, gate):
    """Blocks that add nothing (W2 = 0) leave the recurrence g_l = delta_l + a_l g_{l+1}: the truncated pass's states are those of the
    recurrence in 64 bits, each rounded once; the exact pass goes from one stored state to the next with one rounding each."""
    from paper_2501_17086_b200 import binding as B
    L, d, h, rows = 24, 32, 64, 32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(77)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")
    params = {"W1": rand(L, h, d) / d ** 0.5, "W2": torch.zeros((L, d, h), device="cuda")}
    a = torch.ones((L, d), device="cuda")
    if gate != "one":
        params["a"] = 0.9 + 0.1 * torch.rand((d,) if gate == "shared" else (L, d), generator=gen, device="cuda")
        a = params["a"].expand(L, d)
    delta = rand(L + 1, rows, d)
    ctx = B.Context(B.make_config(block, "f32", L, d, rows, hidden=h, loss=B.LOSS_EVERY_STEP,
                                  gate={"one": B.GATE_ONE, "shared": B.GATE_CHANNEL_SHARED, "per_step": B.GATE_CHANNEL_PER_STEP}[gate]))
    x = ctx.forward(params, rand(rows, d))
    truncated = [ctx.backward(params, k, delta, x) for k in (0, 1)]
    exact = ctx.exact(params, delta, x)
    ctx.sync_status()
    assert ctx.forms["few_rows"] == 4
    ref = delta.double()
    for l in range(L - 1, -1, -1):
        ref[l] += a[l].double() * ref[l + 1]
    for g in truncated:  # half a unit in the last place, and what the sums in 64 bits themselves are off by
        assert bool(((g.double() - ref).abs() <= 2.0 ** -24 * ref.abs() + 2.0 ** -45 * ref.abs().max()).all())
    assert torch.equal(exact[:-1], (a[:, None].double() * exact[1:].double() + delta[:-1].double()).float())


@pytest.mark.parametrize("block", ["mlp", "preln_mlp"])
def test_more_layers_than_the_iterations_have_memory_for_are_exact_in_one_launch(block):
    """The exact pass keeps two layers' products, the iterations all layers'; as many iterations as layers give the same gradients."""
    from paper_2501_17086_b200 import harness
    from paper_2501_17086_b200.workloads import Workload, make_inputs
    w = Workload("t", block, "f32", L=40, d=256, hidden=64, tokens=2, batch=1, seq=1, seed=9899, loss="final_mse")
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    ctx = harness.make_context(w)
    x = ctx.forward(params, inp["x0"])
    delta = harness.loss_delta(w, x, inp)
    exact, all_of_them = ctx.new_grads(), ctx.new_grads()
    g = ctx.exact(params, delta, x, grads=exact)
    assert ctx.forms["few_rows"] == 2
    other = ctx.backward(params, 40, delta, x, grads=all_of_them)
    ctx.sync_status()
    assert ctx.forms["few_rows"] == 2
    bound = 40 * 2 * 2.0 ** -24  # two roundings a layer
    assert float((g - other).norm() / other.norm()) < bound
    for n in exact:
        assert float((exact[n] - all_of_them[n]).norm() / all_of_them[n].norm()) < bound, n


# layers, width, hidden units, block, and whether the iterations of backward(1), backward(4), both with gradients, and the exact pass
# without and with gradients are one launch: the last number of layers that gains by it, and the next
@pytest.mark.parametrize("L,d,h,rows,block,taken", [
    (24, 64, 256, 32, "mlp", "yyyyyy"), (25, 64, 256, 32, "mlp", "nnnnyy"), (24, 64, 1024, 32, "preln_mlp", "yyyyyy"), (25, 64, 1024, 1, "mlp", "nnnnyy"),
    (8, 256, 256, 3, "preln_mlp", "yyyyyy"), (9, 256, 256, 3, "mlp", "nnynyy"), (16, 128, 512, 3, "mlp", "nnynyy"), (17, 128, 512, 3, "mlp", "nnnnyy"),
    (9, 512, 128, 3, "mlp", "nnnnyy"), (73, 256, 256, 3, "mlp", "nnnnyn"), (145, 256, 256, 8, "mlp", "nnnnnn"), (145, 256, 256, 9, "mlp", "nnnnyy"),
    (145, 256, 256, 9, "preln_mlp", "nnnnnn")])
def test_backward_passes_of_deep_stacks_are_one_launch_only_where_that_gains(L, d, h, rows, block, taken):
    from paper_2501_17086_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(81)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")
    params = {"W1": rand(L, h, d) / d ** 0.5, "W2": rand(L, d, h) * (0.5 / (L * h) ** 0.5)}
    ctx = B.Context(B.make_config(block, "f32", L, d, rows, hidden=h))
    x, delta, g = ctx.forward(params, rand(rows, d)), rand(rows, d), ctx.new_states()
    calls = [lambda gr: ctx.backward(params, 1, delta, x, g_all=g, grads=gr), lambda gr: ctx.backward(params, 4, delta, x, g_all=g, grads=gr)] * 2
    calls += [lambda gr: ctx.exact(params, delta, x, g_all=g, grads=gr)] * 2
    got = ""
    for call, with_grads in zip(calls, (0, 0, 1, 1, 0, 1)):
        before = ctx.forms["few_rows"]
        call(ctx.new_grads() if with_grads else None)
        got += "y" if ctx.forms["few_rows"] > before else "n"
    ctx.sync_status()
    assert got == taken


def test_weight_gradients_of_more_layers_than_a_grid_is_deep():
    """The exact pass of any number of layers is one launch; so are its weight gradients, here of 2 x 32769 products (a grid has 65535
    blocks in its third dimension).  Against 64 bits from the pass's own states: sums of two rows and of four units."""
    from paper_2501_17086_b200 import binding as B
    L, d, h, rows = 32769, 4, 4, 2
    gen = torch.Generator(device="cuda")
    gen.manual_seed(79)
    rand = lambda *s: torch.randn(s, generator=gen, device="cuda")
    params = {"W1": rand(L, h, d) / 2, "W2": rand(L, d, h) * (0.5 / L ** 0.5)}
    ctx = B.Context(B.make_config("mlp", "f32", L, d, rows, hidden=h))
    x = ctx.forward(params, rand(rows, d))
    grads = ctx.new_grads()
    g = ctx.exact(params, rand(rows, d), x, grads=grads)
    ctx.sync_status()
    assert ctx.forms["few_rows"] == 2
    z = (x[:-1].double() @ params["W1"].double().mT).requires_grad_()
    act = torch.nn.functional.gelu(z)
    dz, = torch.autograd.grad(act, z, g[1:].double() @ params["W2"].double())
    for got, ref in ((grads["dW1"], dz.mT @ x[:-1].double()), (grads["dW2"], g[1:].double().mT @ act.detach())):
        assert float((got - ref).norm() / ref.norm()) < 8 * 2.0 ** -24


LOWERED = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <cuda_runtime_api.h>
int lowered = 0, limits = 0;
static struct { const void* f; int bytes; } seen[256];
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute attr, int value) {
  if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    int i = 0;
    while (i < limits && seen[i].f != f) ++i;
    if (i == limits && limits < 256) seen[limits++].f = f;
    if (value < seen[i].bytes) ++lowered;
    seen[i].bytes = value;
  }
  typedef cudaError_t (*Fn)(const void*, enum cudaFuncAttribute, int);
  static Fn real = 0;
  if (!real) real = (Fn)dlsym(RTLD_NEXT, "cudaFuncSetAttribute");
  if (!real) real = (Fn)dlsym(dlopen("libcudart.so.12", RTLD_NOW | RTLD_NOLOAD), "cudaFuncSetAttribute");
  return real(f, attr, value);
}
"""

TWO_SIZES = r"""
import ctypes, os
import torch
from paper_2501_17086_b200 import binding as B
stand_in = ctypes.CDLL(os.environ["LD_PRELOAD"])
read = lambda name: ctypes.c_int.in_dll(stand_in, name).value
rand = lambda *s: torch.randn(s, device="cuda")
for L, d, sizes in ((8, 64, (256, 128)), (2, 128, (512, 256))):   # backward 164 and 97 KB a CTA; forward 160 and 94
    for h, rows in zip(sizes, (32, 3)):
        ctx = B.Context(B.make_config("mlp", "f32", L, d, rows, hidden=h))
        params = {"W1": rand(L, h, d) / d ** 0.5, "W2": rand(L, d, h) / h ** 0.5}
        x = ctx.forward(params, rand(rows, d))
        ctx.backward(params, 1, rand(rows, d), x)
        ctx.sync_status()
        assert ctx.forms["few_rows"] == 2
assert read("limits") >= 2 and read("lowered") == 0, (read("limits"), read("lowered"))
print("REFUSED 0")
"""


def test_a_small_stack_does_not_lower_the_memory_limit_of_a_large_one(tmp_path):
    """A kernel's limit of dynamic shared memory belongs to the kernel, whatever thread sets it: a call that set its own size could lower
    it between another thread's set-up and launch, which would then fail.  A stand-in for the runtime's call sees every value set."""
    from test_gpu_refused_clusters import _run_refused
    _run_refused(tmp_path, TWO_SIZES, LOWERED)
