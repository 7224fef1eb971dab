"""Workspace of the float MLP stacks: keeping operands split for the tensor cores may at most treble it or add 64 MiB, up to half of
the device, modes that do not are not charged for it, and a stack runs with less, down to what it takes without."""
import ctypes as C

import pytest
import torch

BLOCKS = ("mlp", "preln_mlp", "relu_mlp", "postln_mlp")


def _config(block, L, d, h, tokens):
    from paper_2501_17086_b200 import binding as B
    return B, B.make_config(block, "f32", L, d, tokens, hidden=h)


def _sizes(monkeypatch, block, L, d, h, tokens):
    B, cfg = _config(block, L, d, h, tokens)
    out = [B.workspace_bytes(cfg)]
    for mode in ("HBP_GEMM_PAIR", "HBP_FORCE_SIMT"):
        with monkeypatch.context() as m:
            m.setenv(mode, "0" if mode == "HBP_GEMM_PAIR" else "1")
            out.append(B.workspace_bytes(cfg))
    return out


@pytest.mark.parametrize("block", BLOCKS)
@pytest.mark.parametrize("L,d,h,tokens", [
    (16, 1024, 4096, 33), (16, 1024, 4096, 40), (16, 1024, 4096, 256), (16, 1024, 4096, 1000), (2, 4096, 16384, 64), (8, 64, 256, 64),
    (3, 68, 68, 200), (12, 520, 1560, 1900), (64, 1024, 4096, 16384), (40, 2048, 8192, 16384), (8, 64, 256, 32), (64, 1024, 4096, 30000),
])
def test_split_operands_are_bounded(monkeypatch, block, L, d, h, tokens):
    most, without, simt = _sizes(monkeypatch, block, L, d, h, tokens)
    assert without == simt <= most <= max(without, min(without + max(2 * without, 64 << 20), 90 << 30))
    # states, dZ and both caches of the block are held in any form (the scratch of a layer group is at least one layer's)
    assert without >= 4 * L * tokens * (d + 2 * h) + 4 * tokens * h
    if tokens <= 32 or d * h > 32 << 20:
        assert most == without
    elif without < 30 << 30:
        assert most > without


@pytest.mark.parametrize("d,h,tokens", [(1024, 4096, 8192), (1024, 1024, 32768), (2048, 8192, 4096)])
def test_scratch_of_a_layer_group_stays_within_6_gib(monkeypatch, d, h, tokens):
    for forms in range(2):  # with planes, without
        a, b = (_sizes(monkeypatch, "preln_mlp", L, d, h, tokens)[forms] for L in (64, 65))
        scratch = a - 64 * (b - a)  # what does not grow with the layers: the group, and partial sums of d channels
        assert 4 << 30 < scratch <= (6 << 30) + 256 * d * 4 + (1 << 16)


@pytest.mark.gpu
@pytest.mark.parametrize("group", ["", "2"])
@pytest.mark.parametrize("block", BLOCKS)
def test_stacks_run_with_less(monkeypatch, block, group):
    from paper_2501_17086_b200 import harness
    from paper_2501_17086_b200.workloads import Workload, make_inputs
    if group:
        monkeypatch.setenv("HBP_LAYER_GROUP", group)
    w = Workload("t", block, "f32", L=5, d=132, hidden=260, tokens=700, batch=1, seq=1, seed=9400, init="small" if block == "postln_mlp" else "")
    most, without, _ = _sizes(monkeypatch, block, w.L, w.d, w.hidden, w.tokens)
    B, cfg = _config(block, w.L, w.d, w.hidden, w.tokens)
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    one_layer = 6 * (w.hidden * 144 + w.d * 320)  # both weights in three planes of two bytes, 132 columns rounded up to 16, 260 to 64

    def shifted(t):  # the same values four bytes past a 16-byte boundary
        out = torch.empty(t.numel() + 4, device="cuda")[1:1 + t.numel()].view(t.shape)
        return out.copy_(t)

    def run(nbytes, pair=True, params=params):
        with monkeypatch.context() as m:
            m.setattr(B, "workspace_bytes", lambda cfg: nbytes)
            if not pair:
                m.setenv("HBP_GEMM_PAIR", "0")
            ctx = harness.make_context(w)
        x = ctx.forward(params, inp["x0"])
        delta = harness.loss_delta(w, x, inp)
        out = [x]
        for exact in (False, True):
            grads = ctx.new_grads()
            out.append(ctx.exact(params, delta, x, grads=grads) if exact else ctx.backward(params, 2, delta, x, grads=grads))
            out += [grads[n] for n in sorted(grads)]
        ctx.sync_status()
        return out, ctx.launches, ctx.forms["gemm_parts"]

    all_layers, launches, products = run(most)
    for layers in (3, 1):  # at a time: the same products, with more split passes between them
        some, more, n = run(most - (w.L - layers) * one_layer)
        assert more > launches and 0 < n <= products  # (batched VJPs of so few layers may split inside)
        assert all(torch.equal(a, b) for a, b in zip(some, all_layers))
    some, _, n = run(most - (w.L - 1) * one_layer, params={k: shifted(t) for k, t in params.items()})
    assert n == products and all(torch.equal(a, b) for a, b in zip(some, all_layers))
    # the operands split inside the kernel: the same arithmetic
    (inside, *n0), (least, *n1) = run(without, pair=False), run(without)
    assert n0 == n1 and n0[0] < launches and n0[1] == 0
    assert all(torch.equal(a, b) and torch.equal(a, c) for a, b, c in zip(inside, least, all_layers))
    h = C.c_void_p()
    ws = torch.empty(without + 256, dtype=torch.uint8, device="cuda")
    assert B.lib.hbp_create(C.byref(cfg), C.c_void_p((ws.data_ptr() + 255) // 256 * 256), without - 1, C.byref(h)) == 5
