"""The LayerNorm of the forward pass where a row takes one, two and four warps (up to 2048, 4096 and 8192 wide), with row counts
that leave its last block part empty and widths that leave a warp's last load part empty, against the oracle."""
import pytest

from oracle import run as orun
from paper_2501_17086_b200.workloads import Workload, make_inputs
from test_gpu_parity import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 3, 5])
@pytest.mark.parametrize("dtype,d", [("bf16", 2048), ("bf16", 2056), ("bf16", 4096), ("bf16", 4104), ("bf16", 8192), ("f32", 2052), ("f32", 4096)])
@pytest.mark.parametrize("block", ["preln_mlp", "postln_mlp"])
def test_wide_rows_match_oracle(block, dtype, d, rows):
    w = Workload("t", block, dtype, L=2, d=d, hidden=64, tokens=rows, batch=1, seq=1, seed=9600 + d + rows,
                 init="small" if block == "postln_mlp" else "")
    inp = make_inputs(w, "cuda")
    # rows far apart in mean and size: one that took another's sums would be off by as much
    for r in range(rows):
        inp["x0"][r] = (inp["x0"][r].float() * (r + 1) + 2 * r).to(inp["x0"].dtype)
    compare(w, run_gpu(w, inp, (1,)), orun.run(w, inp, ks=(1,), grads_for=("exact",)), (1,), ("exact",))
