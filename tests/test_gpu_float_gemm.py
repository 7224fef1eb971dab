"""The float tensor-core GEMM (operands split into two tf32 parts inside the kernel) at the edges of its tiles: rows, columns
and contraction lengths around 32 and 128, every orientation of the operands and every epilogue of the float MLP and decoder
kinds, against the oracle."""
import os

import pytest
import torch

from oracle import run as orun
from paper_2501_17086_b200 import harness
from paper_2501_17086_b200.workloads import Workload, make_inputs
from test_gpu_parity import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block,L,d,h,tokens", [
    ("mlp", 2, 4, 8, 33), ("mlp", 2, 128, 256, 127), ("mlp", 3, 132, 260, 129), ("preln_mlp", 2, 36, 388, 257),
    ("preln_mlp", 2, 260, 124, 1000), ("relu_mlp", 2, 100, 132, 70), ("postln_mlp", 2, 132, 300, 161), ("mlp", 1, 1028, 1032, 40),
])
def test_tile_edges_match_oracle(block, L, d, h, tokens):
    w = Workload("t", block, "f32", L=L, d=d, hidden=h, tokens=tokens, batch=1, seq=1, seed=8000 + d + tokens)
    inp = make_inputs(w, "cuda")
    compare(w, run_gpu(w, inp, (1, L)), orun.run(w, inp, ks=(1, L), grads_for=("exact", L)), (1, L), ("exact", L))


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
    assert torch.equal(finite[0][0], finite[1][0])
    assert torch.equal(finite[0][1].all(dim=1), finite[1][1].all(dim=1))
