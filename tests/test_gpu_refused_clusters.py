"""The one-launch recurrences where the device refuses their cluster launches: a stand-in for the runtime's launch call,
loaded ahead of it in a process of its own, answers "out of resources" to every launch in clusters."""
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


def test_refused_cluster_launches_fall_back_to_one_launch_per_step(tmp_path):
    src, lib = tmp_path / "refuse.c", tmp_path / "librefuse.so"
    src.write_text(REFUSE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-I" + os.path.join(cuda, "include"), str(src), "-o", str(lib), "-ldl"])
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    env.pop("HBP_FORCE_SIMT", None)
    out = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "REFUSED" in out.stdout
