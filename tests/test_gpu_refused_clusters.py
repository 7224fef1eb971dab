"""The one-launch recurrences and the float MLP stacks where the device refuses their cluster launches: a stand-in for the
runtime's launch call, loaded ahead of it in a process of its own, answers "out of resources" to every launch in clusters."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

REFUSE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <cuda_runtime_api.h>
int refused_launches = 0;
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension &&
        c->attrs[i].val.clusterDim.x * c->attrs[i].val.clusterDim.y * c->attrs[i].val.clusterDim.z > 1) {
      ++refused_launches;
      return cudaErrorLaunchOutOfResources;
    }
  typedef cudaError_t (*Fn)(const cudaLaunchConfig_t*, const void*, void**);
  static Fn real = 0;
  if (!real) real = (Fn)dlsym(RTLD_NEXT, "cudaLaunchKernelExC");
  if (!real) real = (Fn)dlsym(dlopen("libcudart.so.12", RTLD_NOW | RTLD_NOLOAD), "cudaLaunchKernelExC");
  return real(c, f, args);
}
"""

CHILD = r"""
import ctypes, os, sys
import torch
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs

refused = ctypes.c_int.in_dll(ctypes.CDLL(os.environ["LD_PRELOAD"]), "refused_launches")
T, B = 7, 40
for block, u in (("gru", 64), ("lstm", 40), ("rnn_tanh", 128), ("rnn_tanh", 100)):
    w = Workload("t", block, "f32", L=T, d=2 * u if block == "lstm" else u, hidden=u if block == "lstm" else 0, in_dim=16,
                 batch=B, tokens=B, seed=9000 + u, loss="every_mse")
    inp = make_inputs(w, "cuda")
    params, xin = harness.params_for(w, inp), harness.rnn_inputs(w, inp)
    outs = []
    for steps in (False, True):
        if steps:
            os.environ["HBP_FORCE_SIMT"] = "1"   # one launch per step
        ctx = harness.make_context(w)
        os.environ.pop("HBP_FORCE_SIMT", None)
        before = refused.value
        x = ctx.forward(params, inp["x0"], xin)
        forward_refused = refused.value - before
        delta = harness.loss_delta(w, x, inp)
        g = ctx.exact(params, delta, x, xin)
        ctx.sync_status()
        if not steps:
            assert forward_refused > 0 and refused.value - before > forward_refused, (block, u, refused.value)
        assert ctx.forms["step"] == 2 * T and not any(ctx.forms[f] for f in ("cell_cluster", "rnn_cluster", "rnn_four_rows")), ctx.forms
        outs.append((x, g))
    # the same per-step kernels on both sides (every cluster refused, theirs too): the same bits
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1]), (block, u)
print("REFUSED", refused.value)
"""


STACKS = r"""
import ctypes, os
import torch
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs

refused = ctypes.c_int.in_dll(ctypes.CDLL(os.environ["LD_PRELOAD"]), "refused_launches")
for block in ("mlp", "preln_mlp", "relu_mlp", "postln_mlp"):
    w = Workload("t", block, "f32", L=3, d=132, hidden=260, tokens=300, batch=1, seq=1, seed=9050, init="small" if block == "postln_mlp" else "")
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    outs = []
    for single in (False, True):
        if single:
            os.environ["HBP_GEMM_PAIR"] = "0"
        ctx = harness.make_context(w)
        os.environ.pop("HBP_GEMM_PAIR", None)
        before = refused.value
        x = ctx.forward(params, inp["x0"])
        delta = harness.loss_delta(w, x, inp)
        got = [x]
        for exact in (False, True):
            grads = ctx.new_grads()
            got.append(ctx.exact(params, delta, x, grads=grads) if exact else ctx.backward(params, 2, delta, x, grads=grads))
            got += [grads[n] for n in sorted(grads)]
        ctx.forward(params, inp["x0"], x_all=x)
        ctx.sync_status()
        # paired CTAs: the first product is refused, and none is asked for again; single CTAs by request: none is asked for
        assert refused.value - before == (0 if single else 1), (block, single, refused.value - before)
        outs.append(got)
    assert all(torch.equal(a, b) for a, b in zip(*outs)), block
print("REFUSED", refused.value)
"""


FEW_ROWS = r"""
import ctypes, os
import torch
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs

refused = ctypes.c_int.in_dll(ctypes.CDLL(os.environ["LD_PRELOAD"]), "refused_launches")
for block in ("mlp", "preln_mlp"):
    w = Workload("t", block, "f32", L=5, d=64, hidden=96, tokens=20, batch=1, seq=1, seed=9060)
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    outs = []
    for single in (False, True):
        if single:
            os.environ["HBP_GEMM_PAIR"] = "0"
        ctx = harness.make_context(w)
        os.environ.pop("HBP_GEMM_PAIR", None)
        before, got = refused.value, []
        for again in range(2):
            x = ctx.forward(params, inp["x0"])
            delta = harness.loss_delta(w, x, inp)
            got.append(x)
            for exact in (False, True):
                grads = ctx.new_grads()
                got.append(ctx.exact(params, delta, x, grads=grads) if exact else ctx.backward(params, 2, delta, x, grads=grads))
                got += [grads[n] for n in sorted(grads)]
        ctx.sync_status()
        assert ctx.forms["few_rows"] == 0
        # the first pass asks once, and no pass asks again; by request none is asked for
        assert refused.value - before == (0 if single else 1), (block, single, refused.value - before)
        outs.append(got)
    assert all(torch.equal(a, b) for a, b in zip(*outs)), block
print("REFUSED", refused.value)
"""


CELL_PRODUCTS = r"""
import ctypes, os
import torch
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs

refused = ctypes.c_int.in_dll(ctypes.CDLL(os.environ["LD_PRELOAD"]), "refused_launches")
for block, u in (("gru", 64), ("lstm", 40), ("rnn_tanh", 100)):
    for T, B, first in ((7, 40, True), (9, 39, False)):
        w = Workload("t", block, "f32", L=T, d=2 * u if block == "lstm" else u, hidden=u if block == "lstm" else 0, in_dim=16,
                     batch=B, tokens=B, seed=9100 + u, loss="every_mse")
        inp = make_inputs(w, "cuda")
        params, xin = harness.params_for(w, inp), harness.rnn_inputs(w, inp)
        outs = []
        for mode in (None, "HBP_GEMM_PAIR", "HBP_FORCE_SIMT"):
            if mode:
                os.environ[mode] = "0" if mode == "HBP_GEMM_PAIR" else "1"
            ctx = harness.make_context(w)
            if mode:
                os.environ.pop(mode)
            x = ctx.forward(params, inp["x0"], xin)
            delta = harness.loss_delta(w, x, inp)
            got, asked = [x], []
            if not first:   # the gradients of the exact pass are the first such product
                grads = ctx.new_grads()
                got += [ctx.exact(params, delta, x, xin, grads=grads)] + [grads[n] for n in sorted(grads)]
            for k in (2, 3, 2):
                before, grads = refused.value, ctx.new_grads()
                got += [ctx.backward(params, k, delta, x, xin, grads=grads)] + [grads[n] for n in sorted(grads)]
                asked.append(refused.value - before)
            ctx.sync_status()
            # the first product is refused, and none is asked for again
            assert asked == ([1, 0, 0] if first and not mode else [0, 0, 0]), (block, T, mode, asked)
            assert ctx.forms["gemm_cell"] == 0
            outs.append(got)
        for other in outs[:2]:   # single CTAs' tf32 products are 1.2e-6 from 64 bits, float sums in any order less
            for a, b in zip(other, outs[2]):
                assert float((a - b).norm() / b.norm()) < 5e-6, (block, T)
print("REFUSED", refused.value)
"""


def _run_refused(tmp_path, child, stand_in=REFUSE):
    src, lib = tmp_path / "refuse.c", tmp_path / "librefuse.so"
    src.write_text(stand_in)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-I" + os.path.join(cuda, "include"), str(src), "-o", str(lib), "-ldl"])
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    for name in ("HBP_FORCE_SIMT", "HBP_GEMM_PAIR"):
        env.pop(name, None)
    out = subprocess.run([sys.executable, "-c", child], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "REFUSED" in out.stdout


def test_refused_cluster_launches_fall_back_to_one_launch_per_step(tmp_path):
    _run_refused(tmp_path, CHILD)


def test_float_stacks_need_no_clusters(tmp_path):
    _run_refused(tmp_path, STACKS)


def test_float_stacks_of_few_rows_take_a_launch_per_product(tmp_path):
    _run_refused(tmp_path, FEW_ROWS)


def test_cell_products_need_no_clusters(tmp_path):
    _run_refused(tmp_path, CELL_PRODUCTS)
