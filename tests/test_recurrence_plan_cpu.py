"""The splits of the one-launch recurrences, looked over on the host: what a plan makes the kernels read and hold stays within
what is there for it."""
import pytest

from paper_2501_17086_b200.build import build_library

# clusters of cs CTAs that a B200 runs at a time, cs = 0..16 (fewer than 148 / cs: a cluster stays within one GPC)
AT_ONCE = [0, 148, 74, 45, 35, 28, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7]


@pytest.fixture(scope="module")
def B():
    build_library()
    from paper_2501_17086_b200 import binding
    return binding


def _config(B, block, dtype, u, rows, nin):
    return B.make_config(block, dtype, 4, 2 * u if block == "lstm" else u, rows, hidden=u if block == "lstm" else 0, in_dim=nin,
                         batch=rows, loss=B.LOSS_EVERY_STEP)


@pytest.mark.parametrize("block", ["gru", "lstm", "rnn_tanh"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_plans_stay_inside_the_packed_weights_and_shared_memory(B, block, dtype):
    for u in (8, 16, 64, 72, 128, 200, 264, 512):
        for rows in (1, 9, 32, 128, 200):
            for nin in (8, 16, 24, 64, 212 if dtype == "f32" else 216):
                for backward in (False, True):
                    p = B.recurrence_plan(_config(B, block, dtype, u, rows, nin), backward, AT_ONCE)
                    if block == "rnn_tanh" and not backward:
                        assert p is None
                        continue
                    assert p is not None, (u, rows, nin, backward)
                    _check(p, u, (u, rows, nin, backward))


@pytest.mark.parametrize("block", ["gru", "lstm", "rnn_tanh"])
def test_every_width_up_to_1536_has_a_split(B, block):
    """Exact backpropagation in one launch throughout; the forward pass of GRU and LSTM but for the sizes at which the per-step
    tiles just fill the chip; beyond 1536 units (96 per CTA, 16 CTAs) neither."""
    declined = []
    for u in range(520, 1537, 8):
        for rows in (1, 8, 32, 64, 100, 128, 300, 1000):
            for backward in (False, True):
                if block == "rnn_tanh" and not backward:
                    continue
                p = B.recurrence_plan(_config(B, block, "f32", u, rows, 64), backward, AT_ONCE)
                if p is None:
                    assert not backward, (u, rows)
                    declined.append((u, rows))
                else:
                    _check(p, u, (u, rows, backward))
    assert all(1032 <= u <= 1184 and rows in (64, 128) for u, rows in declined), declined
    for backward in (False, True):
        assert B.recurrence_plan(_config(B, block, "f32", 1544, 32, 64), backward, AT_ONCE) is None


@pytest.mark.parametrize("block,u,rows,nin,one_launch", [
    ("gru", 1152, 64, 256, False), ("gru", 1152, 56, 256, True), ("gru", 1152, 112, 256, True), ("gru", 1152, 128, 256, False),
    ("gru", 1024, 128, 256, True), ("lstm", 1088, 58, 256, False), ("lstm", 1216, 128, 256, True), ("lstm", 512, 288, 128, False),
    ("lstm", 512, 256, 256, True), ("gru", 512, 288, 32, True),
])
def test_forward_passes_that_are_faster_step_by_step_decline(B, block, u, rows, nin, one_launch):
    """Sizes measured on both sides of the line."""
    assert (B.recurrence_plan(_config(B, block, "f32", u, rows, nin), False, AT_ONCE) is not None) == one_launch


def _check(p, u, what):
    assert p["words_read"] <= p["packed_words"], (what, p)
    assert p["packed_words"] * 16 <= p["pack_bytes"], (what, p)
    assert p["smem"] <= 227 * 1024 and p["threads"] <= 384 and p["cluster"] <= 16, (what, p)
    assert p["cluster"] * p["units_per_cta"] >= u and p["rows"] <= 24, (what, p)
