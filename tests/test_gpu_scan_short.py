"""Scans that a block's ring of loads takes although a thread for each group of channels could: few steps, many channels, one and two
additive streams, every gate that is a stream or a constant, against the recurrence in 64 bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [31, 32, 33, 64, 127])
@pytest.mark.parametrize("rows,d,dtype", [(3, 4, torch.float32), (700, 512, torch.float32), (130, 1000, torch.bfloat16), (600, 1040, torch.bfloat16)])
@pytest.mark.parametrize("every", [False, True])
@pytest.mark.parametrize("gate", ["one", "shared", "per_step"])
def test_short_scans_match_the_recurrence(T, rows, d, dtype, every, gate):
    from paper_2501_17086_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + rows + every)
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda").to(dtype)
    u, a = rand(T, rows, d), None
    if gate != "one":
        a = (0.5 + 0.49 * torch.rand((d,) if gate == "shared" else (T, d), generator=gen, device="cuda")).to(dtype)
    delta = rand(T + 1, rows, d) if every else rand(rows, d)
    need = B.cumsumprod_scratch_bytes(dtype, T, rows, d)
    g = B.cumsumprod(u, delta, a, loss=B.LOSS_EVERY_STEP if every else B.LOSS_FINAL, g=torch.empty((T + 1, rows, d), device="cuda", dtype=dtype),
                     scratch=torch.empty(max(need, 1), dtype=torch.uint8, device="cuda"))
    ref = torch.empty((T + 1, rows, d), dtype=torch.float64, device="cuda")
    ref[T] = (delta[T] if every else delta).double()
    for l in range(T - 1, -1, -1):
        al = 1.0 if a is None else (a if gate == "shared" else a[l]).double()
        ref[l] = al * ref[l + 1] + u[l].double() + (delta[l].double() if every else 0.0)
    # All terms are positive.  Float: the running value is carried in double, so only the result is rounded (2^-24; 1 % for the sums in
    # double).  bf16: the running value is a float, three roundings a step, T of them at most count, and the result (8 bits: 2^-8).
    bound = 1.01 * 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -8 + T * 3 * 2.0 ** -24
    assert bool(((g.double() - ref).abs() <= bound * ref).all())


@pytest.mark.parametrize("block,T", [("gru", 40), ("lstm", 33), ("rnn_tanh", 64)])
@pytest.mark.parametrize("loss", ["every_mse", "final_mse"])
def test_short_recurrences_match_the_oracle(block, T, loss):
    from oracle import run as orun
    from paper_2501_17086_b200.workloads import Workload, make_inputs
    from test_gpu_parity import compare, run_gpu
    w = Workload("t", block, "f32", L=T, d=88 if block == "lstm" else 44, hidden=44 if block == "lstm" else 0, in_dim=8, batch=13, tokens=13,
                 seed=9900 + T, loss=loss)
    inp = make_inputs(w, "cuda")
    gpu = run_gpu(w, inp, (0, 2))
    compare(w, gpu, orun.run(w, inp, ks=(0, 2), grads_for=("exact", 2)), (0, 2), ("exact", 2))
