"""The exponential, reciprocal, sigmoid and tanh that the one-launch recurrences of GRU and LSTM form their gates from, against
80-bit arithmetic and against the library functions, over their whole range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53  # half a unit in the last place, relative


def _values():
    v = [np.linspace(-760.0, 760.0, 400001), np.linspace(-40.0, 40.0, 400001), np.linspace(-2.0, 2.0, 200001)]
    v += [s * np.logspace(-320, 2.9, 40001) for s in (1.0, -1.0)]
    for c in (0.0, 20.0, 36.7368, 354.0, 708.0):  # where a result rounds to one, and where the clamp sets in
        for s in (1.0, -1.0):
            x = np.full(2001, s * c)
            v.append(x + np.arange(-1000, 1001) * np.spacing(x))
    v.append(np.log(2.0) * (np.arange(-1000, 1001) + 0.5))  # ends of the reduced range
    return np.concatenate(v)


def test_gate_functions_over_their_range():
    from paper_2501_17086_b200 import binding as B
    v = _values()
    got = B.gate_math(torch.from_numpy(v).cuda()).cpu().numpy()
    x = np.abs(v).astype(np.longdouble)
    e = np.exp(-np.minimum(x, 708))
    # exp and the reciprocal: within one unit in the last place (2 EPS); the reciprocal's argument as the kernel rounds it
    assert np.max(np.abs(got[:, 0] - e) / e) <= 2 * EPS
    r = 1 / (1 + got[:, 0]).astype(np.longdouble)
    assert np.max(np.abs(got[:, 1] - r) / r) <= 2 * EPS
    # sigmoid: e (2 EPS, weighted e / (1 + e) <= 1/2), the sum 1 + e (EPS), its reciprocal (2 EPS), one product (e: 2 EPS, EPS)
    big, small = 1 / (1 + e), e / (1 + e)
    s, s1 = np.where(v >= 0, big, small), np.where(v >= 0, small, big)
    assert np.max(np.abs(got[:, 2] - s) / s) <= 7 * EPS
    assert np.max(np.abs(got[:, 3] - s1) / s1) <= 7 * EPS
    # tanh = (1 - e) / (1 + e) with e = exp(-2|v|): e's error is absolute in 1 - e (2 EPS), then as above (3 EPS) and one product;
    # its derivative 4 e / (1 + e)^2: e 2, the reciprocal twice 2 x 4, three products
    e2 = np.exp(-np.minimum(2 * x, 708))
    t, d = np.sign(v) * (1 - e2) / (1 + e2), 4 * e2 / (1 + e2) ** 2
    assert np.max(np.abs(got[:, 4] - t)) <= 8 * EPS
    assert np.max(np.abs(got[:, 5] - d) / d) <= 13 * EPS
    # and CUDA's own functions in the same places, away from the clamp (one unit each)
    w = torch.from_numpy(v).cuda()
    lib = torch.exp(-w.abs())
    inside = (w.abs() < 708).cpu().numpy()
    assert np.max(np.abs(got[:, 0] / lib.cpu().numpy() - 1)[inside]) <= 4 * EPS
    assert np.max(np.abs(got[:, 4] - torch.tanh(w).cpu().numpy())) <= 12 * EPS


def test_gate_functions_at_infinities_and_nan():
    from paper_2501_17086_b200 import binding as B
    v = torch.tensor([float("inf"), float("-inf"), float("nan"), 0.0, -0.0, 1e308, -1e308], dtype=torch.float64, device="cuda")
    got = B.gate_math(v).float().cpu().numpy()  # as the states are stored
    assert np.array_equal(got[0], [0, 1, 1, 0, 1, 0]) and np.array_equal(got[5], got[0])
    assert np.array_equal(got[1], [0, 1, 0, 1, -1, 0]) and np.array_equal(got[6], got[1])
    assert np.isnan(got[2]).all()
    assert np.array_equal(got[3], [1, 0.5, 0.5, 0.5, 0, 1]) and np.array_equal(got[4], got[3])
