"""The cases that performance work on this framework is measured by.

A case is one call, or the calls of one training step, that a user of the framework makes through its public entry
points (`binding.Context`, `binding.cumsumprod`, `harness.loss_delta`):

  train     forward pass, loss gradient, Highway-BP backward(k) with parameter gradients: one optimiser step's work
  forward   the forward pass alone (evaluation, or the sequential part of a recurrent training step)
  backward  backward(k) with parameter gradients from the caches of a forward pass made beforehand
  exact     sequential exact backpropagation with parameter gradients, the method's point of comparison
  scan      the reverse diagonal scan on its own

Sizes are those of the repository's workloads (`paper_2501_17086_b200/workloads.py`), ragged sizes between them, and
`draw`'s ranges around them.  Stacks too large to be held three times over on one GPU keep their width, rows and
hidden size and have fewer layers.
"""
import math

import torch

from paper_2501_17086_b200 import binding, harness
from paper_2501_17086_b200.workloads import Workload, make_inputs


def _case(name, do, block, dtype, L, d, tokens, k=0, hidden=0, in_dim=0, n_heads=0, seq=0, loss="final_mse", gamma=0.0):
    return {"name": name, "do": do, "block": block, "dtype": dtype, "L": L, "d": d, "tokens": tokens, "k": k,
            "hidden": hidden, "in_dim": in_dim, "n_heads": n_heads, "seq": seq, "loss": loss, "gamma": gamma}


def _scan(name, dtype, L, rows, d, gate, loss):
    return {"name": name, "do": "scan", "dtype": dtype, "L": L, "tokens": rows, "d": d, "gate": gate, "loss": loss}


def listed():
    return [
        # the smallest stack anybody trains (workload c1): every kernel is tiny, launches and latency are what counts
        _case("tiny_mlp_train", "train", "mlp", "f32", 8, 64, 32, k=4, hidden=256, loss="final_half_sse"),
        # a float residual MLP of middling, ragged size: single precision is what the method is checked in
        _case("float_mlp_train", "train", "preln_mlp", "f32", 12, 520, 1900, k=2, hidden=1560),
        # deep pre-LN bf16 stack (workload c2), a whole training step
        _case("deep_mlp_train", "train", "preln_mlp", "bf16", 64, 1024, 8192, k=2, hidden=4096),
        # the widest stack (workload c5 with 16 of its 128 layers), the backward pass the method is about
        _case("wide_mlp_backward", "backward", "preln_mlp", "bf16", 16, 2048, 16384, k=4, hidden=8192),
        # pre-LN decoder (workload c4), a whole training step
        _case("decoder_train", "train", "preln_transformer", "bf16", 24, 768, 16384, k=4, hidden=3072, n_heads=12, seq=1024),
        # a small decoder on sequences that no tile divides, exact backpropagation layer by layer
        _case("decoder_ragged_exact", "exact", "preln_transformer", "bf16", 6, 512, 8 * 333, hidden=2048, n_heads=8, seq=333),
        # gated tanh RNN over 4096 steps (workload c3): the backward pass, and the sequential forward pass before it
        _case("rnn_backward", "backward", "rnn_tanh", "f32", 4096, 512, 32, k=4, in_dim=256, loss="every_mse"),
        _case("rnn_forward", "forward", "rnn_tanh", "f32", 4096, 512, 32, in_dim=256, loss="every_mse"),
        # GRU on characters (workload g1), a whole training step
        _case("gru_train", "train", "gru", "f32", 256, 512, 128, k=2, in_dim=212, loss="every_mse"),
        # narrow GRU on pixels (workload g2): 64 units, long sequence
        _case("gru_narrow_backward", "backward", "gru", "f32", 1024, 64, 128, k=4, in_dim=4, loss="every_mse"),
        # LSTM on characters (workload l1): exact backpropagation through time
        _case("lstm_exact", "exact", "lstm", "f32", 256, 1024, 128, hidden=512, in_dim=212, loss="every_mse"),
        # the scan on its own, ragged: 11100 channels over 2048 steps with a loss on every state
        _scan("scan_time", "f32", 2048, 37, 300, "shared", "every_mse"),
    ]


# ------------------------------------------------------------------------------------------------- drawn cases
def _log_int(rng, lo, hi, mult=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(mult, int(round(v / mult)) * mult)


_MOST_FLOPS = 4e13  # a drawn case costs no more than the largest listed ones
_MOST_STEPS = 4096 * 32 * 512  # rows x width x steps of a recurrent state


def draw(rng):
    kind = rng.choice(["float_mlp", "mlp", "mlp", "decoder", "rnn", "gru", "lstm", "scan"])
    if kind == "scan":
        dtype = rng.choice(["f32", "bf16"])
        d = _log_int(rng, 32, 2048, 8)
        rows = _log_int(rng, 4, 4096)
        L = min(_log_int(rng, 8, 4096), max(1, 60_000_000 // (d * rows)))
        return {k: v for k, v in _scan("", dtype, L, rows, d, rng.choice(["one", "shared", "shared", "per_step"]),
                                       rng.choice(["final_mse", "every_mse"])).items() if k != "name"}
    k = rng.choice([1, 2, 4])
    if kind == "float_mlp":
        block = rng.choice(["mlp", "preln_mlp", "postln_mlp"])
        d = _log_int(rng, 64, 1024, 4)
        h = _log_int(rng, 2 * d, 4 * d, 4)
        c = _case("", rng.choice(["train", "backward", "exact"]), block, "f32", _log_int(rng, 2, 16), d, _log_int(rng, 32, 4096),
                  k=k, hidden=h, gamma=0.8 if block == "postln_mlp" else 0.0)
        limit = _MOST_FLOPS / 40  # single precision
    elif kind == "mlp":
        block = rng.choice(["preln_mlp", "preln_mlp", "postln_mlp"])
        d = _log_int(rng, 256, 2048, 8)
        c = _case("", rng.choice(["train", "backward", "exact", "forward"]), block, "bf16", _log_int(rng, 4, 64), d,
                  _log_int(rng, 256, 16384), k=k, hidden=_log_int(rng, 2 * d, 4 * d, 8), gamma=0.8 if block == "postln_mlp" else 0.0)
        limit = _MOST_FLOPS
    elif kind == "decoder":
        heads, seq = rng.randint(4, 16), _log_int(rng, 64, 2048)
        batch = max(1, min(_log_int(rng, 1, 32), 16384 // seq))
        c = _case("", rng.choice(["train", "backward", "exact", "forward"]), "preln_transformer", "bf16", _log_int(rng, 2, 24),
                  64 * heads, batch * seq, k=k, hidden=256 * heads, n_heads=heads, seq=seq)
        limit = _MOST_FLOPS
    else:
        block = {"rnn": "rnn_tanh"}.get(kind, kind)
        units = rng.choice([128, 256, 512]) if kind == "rnn" and rng.random() < 0.5 else _log_int(rng, 64, 512, 4)
        B = _log_int(rng, 8, 192)
        T = min(_log_int(rng, 64, 4096 if kind == "rnn" else 1024), _MOST_STEPS // (B * units * (1 if kind == "rnn" else 4)))
        c = _case("", rng.choice(["train", "backward", "exact", "forward"]), block, "f32", T, 2 * units if kind == "lstm" else units, B,
                  k=k, hidden=units if kind == "lstm" else 0, in_dim=_log_int(rng, 4, 256, 4), loss=rng.choice(["every_mse", "every_mse", "final_mse"]))
        limit = None
    while limit and work(c)["flops"] > limit and c["L"] > 2:
        c["L"] -= 1
    while limit and work(c)["flops"] > limit:
        c["tokens"] = c["tokens"] // 2 if c["block"] != "preln_transformer" else c["tokens"] - c["seq"]
    if c["do"] in ("forward", "exact"):
        c["k"] = 0
    return {key: v for key, v in c.items() if key != "name"}


# ------------------------------------------------------------------------------------------------- preparing and running
def _workload(case, seed):
    return Workload("case", case["block"], case["dtype"], L=case["L"], d=case["d"], hidden=case["hidden"], in_dim=case["in_dim"],
                    n_heads=case["n_heads"], head_dim=64 if case["n_heads"] else 0, seq=case["seq"],
                    batch=case["tokens"] // case["seq"] if case["seq"] else case["tokens"], tokens=case["tokens"], seed=seed,
                    loss=case["loss"], gamma=case["gamma"], init="small" if case["block"] == "postln_mlp" else "")


def prepare(case, seed):
    if case["do"] == "scan":
        dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        L, n, d = case["L"], case["tokens"], case["d"]
        loss = binding.LOSS_EVERY_STEP if case["loss"] == "every_mse" else binding.LOSS_FINAL
        u = torch.randn((L, n, d), generator=gen, device="cuda").to(dt)
        delta = torch.randn((L + 1, n, d) if loss else (n, d), generator=gen, device="cuda").to(dt)
        a = None
        if case["gate"] != "one":
            a = (0.9 + 0.099 * torch.rand((d,) if case["gate"] == "shared" else (L, d), generator=gen, device="cuda")).to(dt)
        need = binding.cumsumprod_scratch_bytes(dt, L, n, d)
        return {"do": "scan", "u": u, "delta": delta, "a": a, "loss": loss, "g": torch.empty((L + 1, n, d), device="cuda", dtype=dt),
                "scratch": torch.empty(need, dtype=torch.uint8, device="cuda") if need else None}
    w = _workload(case, seed)
    inp = make_inputs(w, "cuda")
    ctx = harness.make_context(w)
    s = {"do": case["do"], "k": case["k"], "w": w, "inp": inp, "ctx": ctx, "params": harness.params_for(w, inp),
         "xin": harness.rnn_inputs(w, inp), "x_all": ctx.new_states()}
    if case["do"] != "forward":
        s["g_all"], s["grads"] = ctx.new_states(), ctx.new_grads(with_gate=True)
    if case["do"] in ("backward", "exact"):
        ctx.forward(s["params"], inp["x0"], s["xin"], x_all=s["x_all"])
        s["delta"] = harness.loss_delta(w, s["x_all"], inp)
    return s


def run(s):
    do = s["do"]
    if do == "scan":
        return binding.cumsumprod(s["u"], s["delta"], s["a"], loss=s["loss"], g=s["g"], scratch=s["scratch"])
    ctx, params, x_all, xin = s["ctx"], s["params"], s["x_all"], s["xin"]
    if do in ("train", "forward"):
        ctx.forward(params, s["inp"]["x0"], xin, x_all=x_all)
        if do == "forward":
            return x_all
        delta = harness.loss_delta(s["w"], x_all, s["inp"])
    else:
        delta = s["delta"]
    if do == "exact":
        ctx.exact(params, delta, x_all, xin, g_all=s["g_all"], grads=s["grads"])
    else:
        ctx.backward(params, s["k"], delta, x_all, xin, g_all=s["g_all"], grads=s["grads"])
    out = {"g": s["g_all"], "grads": s["grads"]}
    if do == "train":
        out["x"] = x_all
    return out


# ------------------------------------------------------------------------------------------------- the same in 64 bits
def _layers(w, p, X):
    """One function (state, parameters) -> (next state, diagonal of the residual Jacobian) per residual step, with the parameters it
    takes: (function, {gradient name: (tensor, index of its slice or None)})."""
    F = torch.nn.functional

    def mlp(x, W1, W2):
        return F.gelu(x @ W1.T) @ W2.T

    def norm(x):
        return F.layer_norm(x, x.shape[-1:], eps=w.ln_eps)

    def attention(x, Wq, Wk, Wv, Wo):
        y = norm(x).view(w.batch, w.seq, w.d)
        q, k, v = ((y @ W.T).view(w.batch, w.seq, w.n_heads, w.head_dim).transpose(1, 2) for W in (Wq, Wk, Wv))
        future = torch.ones(w.seq, w.seq, dtype=torch.bool, device=x.device).triu(1)
        s = (q @ k.transpose(2, 3) / math.sqrt(w.head_dim)).masked_fill(future, -math.inf)
        return (s.softmax(-1) @ v).transpose(1, 2).reshape(x.shape) @ Wo.T

    def rnn(xt):
        return lambda x, W, U, a: (a * x + torch.tanh(x @ W.T + xt @ U.T), a)

    def gru(xt):
        def step(x, W, U):
            (ur, uz, un), (wr, wz, wn) = (xt @ U.T).chunk(3, -1), (x @ W.T).chunk(3, -1)
            z = torch.sigmoid(uz + wz)
            return z * x + (1 - z) * torch.tanh(un + torch.sigmoid(ur + wr) * wn), z
        return step

    def lstm(xt):
        def step(x, W, U):
            c, h = x.chunk(2, -1)
            i, f, g, o = (xt @ U.T + h @ W.T).chunk(4, -1)
            c = torch.sigmoid(f) * c + torch.sigmoid(i) * torch.tanh(g)
            return torch.cat([c, torch.sigmoid(o) * torch.tanh(c)], -1), torch.cat([torch.sigmoid(f), torch.zeros_like(f)], -1)
        return step

    def post(x, W1, W2):
        y = x + mlp(x, W1, W2)
        return norm(y), (1 - w.gamma) / (y.var(-1, unbiased=False, keepdim=True) + w.ln_eps).sqrt()

    if w.block in ("rnn_tanh", "gru", "lstm"):
        of = {"rnn_tanh": rnn, "gru": gru, "lstm": lstm}[w.block]
        return [(of(X[t].double()), {n: (p[n].double(), None) for n in p}) for t in range(w.L)]
    out = []
    for b in range(w.L):
        if w.block == "preln_transformer":
            out.append((lambda x, *W: (x + attention(x, *W), 1.0), {n: (p[n][b], b) for n in ("Wq", "Wk", "Wv", "Wo")}))
        whole = {"mlp": lambda x, *W: (x + mlp(x, *W), 1.0), "postln_mlp": post}.get(w.block, lambda x, *W: (x + mlp(norm(x), *W), 1.0))
        out.append((whole, {n: (p[n][b], b) for n in ("W1", "W2")}))
    return out


def exact(case, seed):
    """What `run` returns, from the same inputs, with every operation in 64 bits: each layer's vector-Jacobian product is
    automatic differentiation of the layer less its residual part, and the scan is its recurrence."""
    if case["do"] == "scan":
        s = prepare(case, seed)
        delta, every, L = s["delta"].double(), case["loss"] == "every_mse", case["L"]
        g = torch.empty(s["g"].shape, dtype=torch.float64, device="cuda")
        g[L] = delta[L] if every else delta
        for l in range(L - 1, -1, -1):
            a = 1.0 if s["a"] is None else (s["a"] if s["a"].dim() == 1 else s["a"][l]).double()
            g[l] = a * g[l + 1] + s["u"][l].double() + (delta[l] if every else 0.0)
        return g
    w = _workload(case, seed)
    inp = make_inputs(w, "cuda")
    params = harness.params_for(w, inp)
    layers = _layers(w, params, inp.get("X"))
    n = len(layers)
    x = torch.empty((n + 1, w.tokens, w.d), dtype=torch.float64, device="cuda")
    x[0] = inp["x0"].double()
    keep = []  # diagonals of the residual Jacobians, None where they are one
    with torch.no_grad():
        for l, (f, p) in enumerate(layers):
            x[l + 1], a = f(x[l], *(t.double() for t, _ in p.values()))
            keep.append(a)
    if case["do"] == "forward":
        return x
    delta = torch.zeros_like(x)
    if w.loss == "every_mse":
        delta[1:] = (x[1:] - inp["Y"].double()) * (2.0 / (w.L * w.batch * w.d))
    else:
        delta[n] = (x[n] - inp["y"].double()) * (1.0 if w.loss == "final_half_sse" else 2.0 / (w.tokens * w.d))
    grads = {"d" + name: torch.zeros(t.shape, dtype=torch.float64, device="cuda") for name, t in params.items()}

    def vjp(l, v, state=True, weights=False):
        f, p = layers[l]
        at = x[l].clone().requires_grad_(state)
        ws = [t.double().clone().requires_grad_(weights) for t, _ in p.values()]
        got = list(torch.autograd.grad(f(at, *ws)[0], ([at] if state else []) + (ws if weights else []), v))
        back = got.pop(0) if state else None
        for (name, (_, i)), t in zip(p.items(), got):
            (grads["d" + name] if i is None else grads["d" + name][i]).add_(t)
        return back

    g = torch.empty_like(x)
    g[n] = delta[n]
    if case["do"] == "exact":
        for l in range(n - 1, -1, -1):
            g[l] = delta[l] + vjp(l, g[l + 1], weights=True)
    else:
        for l in range(n - 1, -1, -1):
            g[l] = delta[l] + keep[l] * g[l + 1]
        for _ in range(min(case["k"], n)):
            new = delta[n]
            for l in range(n):  # the products of the old estimate first: g[l] is not read again
                g[l] = vjp(l, g[l + 1]) - keep[l] * g[l + 1]
            for l in range(n - 1, -1, -1):
                new = delta[l] + keep[l] * new + g[l]
                g[l] = new
        for l in range(n):
            vjp(l, g[l + 1], state=False, weights=True)
    out = {"g": g, "grads": grads}
    if case["do"] == "train":
        out["x"] = x
    return out


# ------------------------------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    es = 4 if case["dtype"] == "f32" else 2
    L, n, d = case["L"], case["tokens"], case["d"]
    if case["do"] == "scan":
        every = case["loss"] == "every_mse"
        tensors = L + (L + 1) + ((L + 1) if every else 1)
        gate = {"one": 0, "shared": d, "per_step": L * d}[case["gate"]]
        return {"bytes": (tensors * n * d + gate) * es, "flops": (2 + every) * L * n * d}
    h, nin, block, do, k = case["hidden"], case["in_dim"], case["block"], case["do"], case["k"]
    steps = 2 * L if block == "preln_transformer" else L
    k = min(k, steps)
    # per row of a state and step (decoder block): flops of the forward pass, of one VJP, and of the parameter pass
    # given the VJP's intermediate results (exact) or forming them again (from the final estimate)
    if block == "rnn_tanh":
        weights, fwd, vjp, grad, again = d * (d + nin), 2 * d * (d + nin), 2 * d * d, 2 * d * (d + nin), 0
    elif block == "gru":
        weights, fwd, vjp, grad, again = 3 * d * (d + nin), 6 * d * (d + nin), 6 * d * d, 6 * d * (d + nin), 0
    elif block == "lstm":
        weights, fwd, vjp, grad, again = 4 * h * (h + nin), 8 * h * (h + nin), 8 * h * h, 8 * h * (h + nin), 0
    elif block == "preln_transformer":
        att = case["seq"] * d  # one causal S x S x head_dim product over all heads, per token
        weights = L * (4 * d * d + 2 * d * h)
        fwd, vjp, grad, again = 8 * d * d + 2 * att + 4 * d * h, 8 * d * d + 5 * att + 4 * d * h, 8 * d * d + 4 * d * h, 2 * d * d + 5 * att + 2 * d * h
    else:
        weights, fwd, vjp, grad, again = L * 2 * d * h, 4 * d * h, 4 * d * h, 4 * d * h, 2 * d * h
    per = {"forward": fwd, "train": fwd + k * vjp + grad + again, "backward": k * vjp + grad + again, "exact": vjp + grad}[do]
    states = (steps + 1) * n * d * es
    inputs = L * n * nin * es
    deltas = (states if case["loss"] == "every_mse" else n * d * es)
    moved = weights * es + inputs + states  # forward: states written; backward: states read
    if do != "forward":
        moved += weights * 4 + states + deltas
    return {"bytes": moved, "flops": per * n * L}


def tolerance(case):
    # Four times what a path differs by from itself evaluated in 64 bits (bf16: 2.6e-3 on the states' gradients,
    # 4e-3 in the exact pass; float: up to 2.7e-6 in the parameter gradients; a scan's bf16 output: one rounding).
    if case["dtype"] == "bf16":
        return {"rel": 8e-3 if case["do"] == "scan" else 1.6e-2}
    if case["do"] == "scan":
        return {"rel": 1e-6}
    # The long gated tanh RNN amplifies the rounding of its forward pass: two evaluations in 64 bits with their sums
    # in another order differ by 2.8e-5 in the exact gradient and by a few 1e-6 in the truncated one.
    if case["block"] == "rnn_tanh" and case["do"] != "forward":
        return {"rel": 1.2e-4 if case["do"] == "exact" else 4e-5}
    return {"rel": 1e-5}
