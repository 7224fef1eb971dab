"""The time scan that streams through a ring of TMA boxes, where its stages and its rows of 512 bytes end: step counts around
the multiples of a stage, rows that fill a block in part, one and two additive streams, against the recurrence in 64 bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _reference(u, delta, a, every):
    L, g = u.shape[0], [None] * (u.shape[0] + 1)
    g[L] = delta[L] if every else delta
    for l in range(L - 1, -1, -1):
        g[l] = a * g[l + 1] + (u[l] + (delta[l] if every else 0.0))
    return torch.stack(g)


@pytest.mark.parametrize("T", [32, 39, 64, 65, 127, 288, 1031])
@pytest.mark.parametrize("rows,d,dtype", [(7, 12, torch.float32), (32, 140, torch.float32), (5, 24, torch.bfloat16)])
@pytest.mark.parametrize("every", [False, True])
def test_ring_scan_matches_the_recurrence(T, rows, d, dtype, every):
    from paper_2501_17086_b200 import binding as B
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + rows + every)
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda").to(dtype)
    u, a = rand(T, rows, d), (0.5 + 0.49 * torch.rand((d,), generator=gen, device="cuda")).to(dtype)
    delta = rand(T + 1, rows, d) if every else rand(rows, d)
    need = B.cumsumprod_scratch_bytes(dtype, T, rows, d)
    g = B.cumsumprod(u, delta, a, loss=B.LOSS_EVERY_STEP if every else B.LOSS_FINAL, g=torch.empty((T + 1, rows, d), device="cuda", dtype=dtype),
                     scratch=torch.empty(max(need, 1), dtype=torch.uint8, device="cuda"))
    ref = _reference(u.double(), delta.double(), a.double(), every)
    # All terms are positive.  Float: u + delta rounded once, the result once, the running value carried in double.  bf16: the
    # running value is a float, three roundings a step that a step multiplies by a < 0.995 (200 of them count), and the result (8 bits: 2^-8).
    bound = 2.1 * 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -8 + 200 * 3 * 2.0 ** -24
    assert float(((g.double() - ref).abs() / ref).max()) <= bound


def test_ring_scan_carries_what_is_not_finite():
    from paper_2501_17086_b200 import binding as B
    T, rows, d = 100, 3, 32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    u = torch.randn((T, rows, d), generator=gen, device="cuda")
    u[50, 0, 3], u[90, 1, 4], u[10, 2, 5], u[10, 2, 6] = float("inf"), float("-inf"), float("nan"), 3.0e38
    u[9, 2, 6], u[70, 0, 7], u[60, 0, 7] = 3.0e38, float("inf"), float("-inf")
    u[40, 1, 8:16] = torch.finfo(torch.float32).tiny / 4
    a = torch.full((d,), 0.9, device="cuda")
    a[5:6] = 0.0
    delta = torch.zeros((rows, d), device="cuda")
    need = B.cumsumprod_scratch_bytes(torch.float32, T, rows, d)
    g = B.cumsumprod(u, delta, a, loss=B.LOSS_FINAL, g=torch.empty((T + 1, rows, d), device="cuda"),
                     scratch=torch.empty(max(need, 1), dtype=torch.uint8, device="cuda"))
    ref = _reference(u.double(), delta.double(), a.double(), False).float()
    torch.testing.assert_close(g, ref, rtol=2.1 * 2.0 ** -24, atol=0.0, equal_nan=True)
