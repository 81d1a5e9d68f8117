"""What is timed: global rounds of distributed sign momentum as a training program runs them.

A case is one problem (a parameter layout, n workers, tau local steps, a base optimizer, a global step) and the way a
program drives it:

- ``round``: the program has written every worker's gradient into the library's buffers (``grad_view``); a pass is
  tau x ``local_step`` and ``global_step``.  What a training loop asks of the library besides its own backward passes.
- ``synthetic``: a pass is ``synthetic_round(with_stats=True)``: the built-in gradient generator in the place of the
  backward pass, and the round's statistics read on the host.
- ``host``: the gradients lie in pinned host memory; a pass is tau x ``local_step_host_grads`` and ``global_step``.
- ``noalloc``: a pass is ``dsm_global_step_noalloc`` on the caller's own x, m and replicas.

Outputs are the state itself (x, m, the replicas, the base optimizers' states, the global second moment, the round's
statistics), as views of the arena.
"""
import ctypes
import math
import types

import torch

from paper_2411_17866_gb300 import dsm

VOCAB, CONTEXT = 50257, 1024
GLOBALS = {"sign": dsm.GLOBAL_SIGN_MOMENTUM, "slowmo": dsm.GLOBAL_SLOWMO, "signed_slowmo": dsm.GLOBAL_SIGNED_SLOWMO,
           "lookahead": dsm.GLOBAL_LOOKAHEAD, "adamw": dsm.GLOBAL_ADAMW}
SIGNS = {"sign": dsm.SIGN, "rsign_zero": dsm.RSIGN_ZERO, "rsign_pm": dsm.RSIGN_PM}
# the most worker-elements of one problem that exact() evaluates in 64 bits
EXACT_MOST = 600_000_000


def _case(name, layout, a, b, n, tau, base="adamw", grads="f32", glob="sign", sign="sign", path="round", fused=True,
          restart=False):
    return {"name": name, "layout": layout, "a": a, "b": b, "n": n, "tau": tau, "base": base, "grads": grads,
            "global": glob, "sign": sign, "path": path, "fused": fused, "restart": restart}


def listed():
    return [
        # a two-layer MLP trained on four workers, options as by default: latency and launches
        _case("mlp-4.5k-n4", "mlp", 32, 64, 4, 4, fused=False),
        # the smallest measured workload, as the README runs it: generator, statistics on the host
        _case("flat-1m-synthetic-n4", "flat", 1 << 20, 0, 4, 4, path="synthetic"),
        # GPT-2 small on four workers, twelve local steps a round
        _case("gpt2-124m-adamw-n4", "gpt2", 12, 768, 4, 12),
        # GPT-2 medium on eight workers with bf16 gradients: the largest state here (45 GB)
        _case("gpt2-355m-adamw-bf16-n8", "gpt2", 24, 1024, 8, 2, grads="bf16"),
        # the width of GPT-2 large with SGD-momentum and the randomized sign, eight workers
        _case("gpt2-184m-sgdm-rsign-n8", "gpt2", 6, 1280, 8, 2, base="sgdm", sign="rsign_zero"),
        # a transformer whose widths, bias tables and learned scalars are odd, options as by default
        _case("odd-9m-adamw-n4", "odd", 9, 289, 4, 2, fused=False),
        # the same kind of layout in a fused round, larger, with bf16 gradients
        _case("odd-30m-adamw-bf16-n4", "odd", 12, 451, 4, 2, grads="bf16"),
        # sixteen workers that synchronise after every step, randomized sign
        _case("flat-16m-sgdm-rsign-n16", "flat", 16_000_000, 0, 16, 1, base="sgdm", sign="rsign_zero"),
        # many workers on a small model, SlowMo
        _case("mlp-283k-slowmo-n32", "mlp", 784, 301, 32, 2, glob="slowmo", fused=False),
        # global AdamW, the base optimizer restarted every round
        _case("gpt2-16m-gadamw-bf16-n6", "gpt2", 4, 256, 6, 2, grads="bf16", glob="adamw", restart=True),
        # a plugin inside a framework that owns the memory: the global step on its buffers
        _case("noalloc-gpt2-3m-n4", "gpt2", 2, 64, 4, 1, path="noalloc"),
        # gradients from pinned host memory
        _case("host-gpt2-16m-adamw-bf16-n4", "gpt2", 4, 256, 4, 2, grads="bf16", path="host"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        layout = rng.choice(["flat", "mlp", "odd", "gpt2", "odd"])
        if layout == "flat":
            a, b = log_int(1_000, 40_000_000), 0
        elif layout == "mlp":
            a, b = log_int(8, 4000), log_int(8, 4000)
        elif layout == "odd":
            a, b = rng.randint(1, 16), log_int(9, 600)
        else:
            a, b = rng.randint(1, 8), 8 * log_int(4, 48)
        path = rng.choice(["round"] * 6 + ["noalloc"] * 2 + ["synthetic", "host"])
        n = log_int(1, 64)
        base = rng.choice(["adamw", "adamw", "sgdm"])
        glob = rng.choice(["sign"] * 5 + ["slowmo", "signed_slowmo", "lookahead", "adamw"])
        if path == "noalloc" and glob == "adamw":
            glob = "slowmo"
        sign = rng.choice(["sign", "sign", "rsign_zero", "rsign_pm"]) if glob == "sign" else "sign"
        c = _case("", layout, a, b, n, 1 if path == "noalloc" else rng.choice([1, 2, 4, 12]), base,
                  rng.choice(["f32", "bf16"]), glob, sign, path, rng.random() < 0.5,
                  path == "round" and rng.random() < 0.15)
        del c["name"]
        d = sum(t.numel for t in _layout(c))
        if n * d <= 300_000_000 and (path != "host" or n * d <= 60_000_000):
            return c


def _layout(case):
    """The tensor list, (numel, grad_scale, kind, wd) each: weights, then their biases."""
    a, b = case["a"], case["b"]
    w, s = 1e-3, 1e-4

    def weight(k):
        return dsm.LayoutEntry(k, w, dsm.KIND_WEIGHT, 1)

    def bias(k):
        return dsm.LayoutEntry(k, s, dsm.KIND_BIAS, 0)

    def norm(k):
        return [dsm.LayoutEntry(k, s, dsm.KIND_LN_W, 1), dsm.LayoutEntry(k, s, dsm.KIND_LN_B, 1)]

    if case["layout"] == "flat":
        return [weight(a)]
    if case["layout"] == "mlp":    # a -> b -> b/2 -> 10
        h = max(1, b // 2)
        return [weight(a * b), bias(b), weight(b * h), bias(h), weight(h * 10), bias(10)]
    if case["layout"] == "gpt2":   # a layers of width b
        t = [weight(VOCAB * b), weight(CONTEXT * b)]
        for _ in range(a):
            t += norm(b) + [weight(3 * b * b), bias(3 * b), weight(b * b), bias(b)]
            t += norm(b) + [weight(4 * b * b), bias(4 * b), weight(4 * b * b), bias(b)]
        return t + norm(b)
    t = [bias(1), weight(1009 * b)]  # a layers of width b: a learned scalar, a relative position table per layer
    for _ in range(a):
        t += norm(b) + [weight(3 * b * b), bias(3 * b), weight(507), weight(b * b), bias(b), bias(1)]
        t += norm(b) + [weight(4 * b * b), bias(4 * b), weight(4 * b * b), bias(b)]
    return t + norm(b) + [weight(b * 10), bias(10)]


def _hparams(case, seed):
    sgdm = case["base"] == "sgdm"
    flags = (dsm.FLAG_FUSED_ROUND if case["fused"] else 0) | (dsm.FLAG_RESET_LOCAL_STATE if case["restart"] else 0)
    return types.SimpleNamespace(
        base=dsm.BASE_SGDM if sgdm else dsm.BASE_ADAMW, lr=1e-2 if sgdm else 6e-4, b1=0.9, b2=0.95, eps=1e-8,
        wd=0.0 if sgdm else 0.1, mu=0.9, g_b1=0.9, g_b2=0.99, g_eta=1e-3, g_wd=0.1, sign_mode=SIGNS[case["sign"]],
        rsign_B=1e-2, grad_dtype=dsm.BF16 if case["grads"] == "bf16" else dsm.F32, flags=flags, seed=seed & 0xFFFFFFFF,
        global_mode=GLOBALS[case["global"]], g_eps=1e-8)


def _x0(d, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(d, device="cuda", generator=g) * 0.02


def _grads(case, d, seed):
    """Every worker's gradient: a common part and the worker's own, in the gradient type."""
    g = torch.Generator("cuda").manual_seed(seed + 1_000_003)
    dt = torch.bfloat16 if case["grads"] == "bf16" else torch.float32
    common = torch.randn(d, device="cuda", generator=g)
    for _ in range(case["n"]):
        own = torch.randn(d, device="cuda", generator=g)
        yield own.mul_(0.5).add_(common).mul_(1e-3).to(dt)


def _replicas(case, d, stride, x, seed):
    """Worker models a few local steps away from x, for the global step on the caller's buffers."""
    r = torch.zeros(case["n"], stride, device="cuda")
    lr = _hparams(case, seed).lr
    for i, g in enumerate(_grads({**case, "grads": "f32"}, d, seed)):
        r[i, :d] = x - lr * 1e3 * g
    return r


def _state_views(run, case):
    """Views of the state's buffers in the arena.  Each buffer is found by the values that a write through the library
    puts at its start (buffers start on 256-byte boundaries); the values there before are written back."""
    rows = run.arena[: run.nbytes // 256 * 256].view(torch.float32).view(-1, 64)
    buffers = {"x": dsm.BUF_X, "m": dsm.BUF_M}
    if not case["fused"]:
        buffers["replicas"] = dsm.BUF_REPLICA      # after a fused round every worker's model is x itself
    if not case["restart"]:
        buffers["opt_m"] = dsm.BUF_OPT_M           # with a restart the states between rounds are zero
        if case["base"] == "adamw":
            buffers["opt_v"] = dsm.BUF_OPT_V
    if case["global"] == "adamw":
        buffers["global_v"] = dsm.BUF_GLOBAL_V
    k = min(run.d, 3)
    mark = torch.tensor([-1.7320508e30, 3.1415926e30, -2.7182818e30][:k], device="cuda")
    views = {}
    for name, which in buffers.items():
        was = run.read(which, count=k, out=torch.empty(k, device="cuda"))
        run.write(which, mark)
        at = int(torch.nonzero((rows[:, 0] == mark[0]) & (rows[:, k - 1] == mark[k - 1]))[0])
        run.write(which, was)
        flat = rows.view(-1)[at * 64:]
        views[name] = flat[: run.d] if name in ("x", "m", "global_v") else \
            flat.as_strided((run.n, run.d), (run.d_stride, 1))
    off = dsm.dsm_stats_ptr(run.h) - run.arena.data_ptr()
    return {**views, **_stats_views(run.arena[off:off + 48 * run.num_tensors].view(run.num_tensors, 48))}


def _stats_views(rows):
    return {"stats_sums": rows.view(torch.float64)[:, :2], "stats_counts": rows.view(torch.int64)[:, 2:]}


def prepare(case, seed):
    layout, hp = _layout(case), _hparams(case, seed)
    d = sum(t.numel for t in layout)
    s = types.SimpleNamespace(path=case["path"], tau=case["tau"])
    x0 = _x0(d, seed)
    if case["path"] == "noalloc":
        stride = -(-d // 64) * 64
        s.x, s.m, s.n, s.stride, s.round = x0, torch.zeros(d, device="cuda"), case["n"], stride, 0
        s.replicas = _replicas(case, d, stride, x0, seed)
        s.layout, s.hp, s.gamma = dsm.make_layout(layout), dsm.make_hparams(hp), hp.lr
        stats = torch.zeros(len(layout), 48, dtype=torch.uint8, device="cuda")
        s.stats = stats
        s.outputs = {"x": s.x, "m": s.m, "replicas": s.replicas[:, :d], **_stats_views(stats)}
        return s
    s.run = dsm.DistributedSignMomentum(layout, case["n"], case["tau"], hp, x0=x0)
    s.outputs = _state_views(s.run, case)
    if case["path"] == "host":
        dt = torch.bfloat16 if case["grads"] == "bf16" else torch.float32
        s.grads = torch.empty(case["n"], d, dtype=dt, pin_memory=True)
        for i, g in enumerate(_grads(case, d, seed)):
            s.grads[i].copy_(g)
        s.copies = torch.cuda.Stream()
    elif case["path"] == "round":
        for i, g in enumerate(_grads(case, d, seed)):
            s.run.grad_view(i).copy_(g)
    return s


def run(s):
    if s.path == "noalloc":
        dsm.dsm_global_step_noalloc(s.layout, s.n, s.hp, s.gamma, s.round, s.x.data_ptr(), s.m.data_ptr(),
                                    s.replicas.data_ptr(), s.stride, s.stats.data_ptr(), stats_is_device=True)
        s.round += 1
    elif s.path == "synthetic":
        s.run.synthetic_round(with_stats=True)
    else:
        for _ in range(s.tau):
            if s.path == "host":
                s.run.local_step_host_grads(s.grads, copy_stream=s.copies)
            else:
                s.run.local_step()
        s.run.global_step()
    return s.outputs


def work(case):
    """Bytes: every local step reads the worker's model, states and gradient and writes model and states (the
    generator writes the gradient first); the global step reads x, m and the replicas and writes x, m and, where the
    workers do not restart from x itself, the replicas.  In a fused round with up to eight workers the last local
    step's models are not written and not read again; a restarted optimizer's states are neither read in the first
    step of a round nor, fused, written in the last one.  Every byte of host gradients is counted once."""
    d = sum(t.numel for t in _layout(case))
    n, tau = case["n"], case["tau"]
    globals_ = 3 if case["global"] == "adamw" else 2
    if case["path"] == "noalloc":
        return {"bytes": float(d * (8 * n + 16)), "flops": float(d * (8 * n + 12))}
    states = 2 if case["base"] == "adamw" else 1
    g = 2 if case["grads"] == "bf16" else 4
    step = 8 + 8 * states + g + (g if case["path"] == "synthetic" else 0)
    per = n * tau * step + 8 * globals_ + n * 8
    if case["restart"]:
        per -= 4 * n * states
    if case["fused"]:
        per -= 4 * n + (n - 1) * 4       # no replica is written back; the round's first step reads x once
        if n <= 8:
            per -= 8 * n                 # the last step's models stay on the chip
            per -= 4 * n * states if case["restart"] else 0
    flops = n * tau * (18 if states == 2 else 4) + 8 * n + 12
    return {"bytes": float(d * per), "flops": float(d * flops)}


def tolerance(case):
    # all arithmetic is fp32, one rounding per operation, summed in worker order.  Against 64 bits the momentum and the
    # statistics are off most: they hold x - x_i, a difference of nearly equal numbers (1.4e-5 for m at most).  The
    # global AdamW step divides by the root of its square, and x is off by 7e-5 where that is near zero.
    rel = 3e-4 if case["global"] == "adamw" else 6e-5
    return {"rel": rel, "max": 40 * rel}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------

_M32 = 0xFFFFFFFF


def _signed(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _finalise(z):
    z = (z ^ _shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _uniform(seed, stream, idx, e):
    """The generator's 24-bit draws of elements e: two of each SplitMix64 output."""
    gold = 0x9E3779B97F4A7C15
    key = int(_finalise(torch.tensor(_signed(seed + (1 + (stream << 40) + idx) * gold))))
    h = _finalise(key + ((e >> 1) + 1) * _signed(gold))
    return torch.where((e & 1) == 1, (h >> 16) & 0xFFFFFF, (h >> 40) & 0xFFFFFF).double() * 2.0 ** -24


def _synthetic_grad(case, hp, scale, e, step, worker):
    s, s2 = scale.double(), (scale * 0.1).double()   # fp32 scales
    g = s * (_uniform(hp.seed, 0, step, e) - 0.5)
    g = (g.float() + (s2 * (_uniform(hp.seed, 1, worker, e) - 0.5)).float())
    return (g.bfloat16() if case["grads"] == "bf16" else g).double()


def _philox_unit(e, k0, k1):
    """Word e mod 4 of Philox4x32-10 with counter e / 4, as a 24-bit uniform."""
    c = [(e >> 2) & _M32, (e >> 2) >> 32, torch.zeros_like(e), torch.zeros_like(e)]

    def mul(a, v):
        return ((a * (v >> 16) + ((a * (v & 0xFFFF)) >> 16)) >> 16), (_signed(a) * v) & _M32

    for r in range(10):
        hi0, lo0 = mul(0xD2511F53, c[0])
        hi1, lo1 = mul(0xCD9E8D57, c[2])
        a, b = (k0 + r * 0x9E3779B9) & _M32, (k1 + r * 0xBB67AE85) & _M32
        c = [hi1 ^ c[1] ^ a, lo1, hi0 ^ c[3] ^ b, lo0]
    w = e & 3
    word = torch.where(w == 0, c[0], torch.where(w == 1, c[1], torch.where(w == 2, c[2], c[3])))
    return (word >> 8).double() * 2.0 ** -24


def _f32(v):
    return ctypes.c_float(v).value


def exact(case, seed):
    """One round from the first state, every operation in 64 bits.  The counts of the statistics are not computed:
    near zero a sign depends on the last bit."""
    layout, hp = _layout(case), _hparams(case, seed)
    n, tau, d = case["n"], case["tau"], sum(t.numel for t in layout)
    if n * d > EXACT_MOST:
        return None
    numels = torch.tensor([t.numel for t in layout], device="cuda")
    wd = torch.repeat_interleave(torch.tensor([float(t.wd != 0) for t in layout], device="cuda").double(), numels)
    tensor = torch.repeat_interleave(torch.arange(len(layout), device="cuda"), numels)
    e = torch.arange(d, device="cuda")
    # hyper-parameters and the scalars derived from them are fp32 values
    lr, eta, lam = _f32(hp.lr), _f32(hp.g_eta), _f32(hp.g_wd)
    x32 = _x0(d, seed)
    x = x32.double()
    m, v = torch.zeros_like(x), torch.zeros_like(x)
    X = torch.empty(n, d, dtype=torch.float64, device="cuda")
    om, ov = torch.zeros_like(X), torch.zeros_like(X) if case["base"] == "adamw" else None
    if case["path"] == "noalloc":
        X[:] = _replicas(case, d, d, x32, seed)
    else:
        scale = torch.repeat_interleave(torch.tensor([t.grad_scale for t in layout], device="cuda"), numels)
        given = None if case["path"] == "synthetic" else _grads(case, d, seed)
        for i in range(n):
            X[i] = x
            own = None if given is None else next(given).double()
            for k in range(tau):
                g = own if own is not None else _synthetic_grad(case, hp, scale, e, k, i)
                if ov is None:
                    om[i].mul_(_f32(hp.mu)).add_(g)
                    X[i].sub_(om[i], alpha=lr)
                    continue
                b1, b2 = _f32(hp.b1), _f32(hp.b2)
                om[i].mul_(b1).add_(g, alpha=_f32(1 - b1))
                ov[i].mul_(b2).addcmul_(g, g, value=_f32(1 - b2))
                step = om[i] / _f32(1 - b1 ** (k + 1)) / ((ov[i] / _f32(1 - b2 ** (k + 1))).sqrt_() + _f32(hp.eps))
                X[i].sub_(step.addcmul_(wd, X[i], value=_f32(hp.wd)), alpha=lr)
    delta = torch.zeros_like(x)
    for i in range(n):
        delta += x - X[i]
    delta /= n
    drift = torch.zeros_like(x)
    for i in range(n):
        drift += (x - X[i] - delta) ** 2
    sums = torch.zeros(len(layout), 2, dtype=torch.float64, device="cuda")
    sums[:, 0].index_add_(0, tensor, delta ** 2)
    sums[:, 1].index_add_(0, tensor, drift)
    b1, b2, mode = _f32(hp.g_b1), _f32(hp.g_b2), case["global"]
    c1, c2 = _f32((1 - b1) / lr), _f32((1 - b2) / lr)
    if mode == "sign":
        u = c1 * delta
        s = torch.sign(u)
        if case["sign"] != "sign":
            p = (u.abs() / _f32(hp.rsign_B)).clamp_(max=1.0)
            r = _philox_unit(e, hp.seed & _M32, 0)
            s = torch.where(r < p, s, 0.0 * s) if case["sign"] == "rsign_zero" else \
                torch.where(r < 0.5 + 0.5 * p, s, -s)
        x = x - _f32(eta * lr) * (s + lam * wd * x)
        m = c2 * delta
    elif mode == "slowmo":
        m = _f32(1 / lr) * delta
        x = x - _f32(eta * lr) * m
    elif mode == "signed_slowmo":
        x = x - _f32(eta * lr) * c1 * torch.sign(delta)
        m = c2 * delta
    elif mode == "lookahead":
        x = x - _f32(eta * lr) * c1 * delta
        m = c2 * delta
    else:
        g = _f32(1 / lr) * delta
        m, v = _f32(1 - b1) * g, _f32(1 - b2) * g * g
        x = x - eta * (m / _f32(1 - b1) / ((v / _f32(1 - b2)).sqrt_() + _f32(hp.g_eps)) + lam * wd * x)
    out = {"x": x, "m": m, "stats_sums": sums, "stats_counts": None}
    if case["path"] == "noalloc" or not case["fused"]:
        out["replicas"] = x.expand(n, d)
    if case["path"] != "noalloc" and not case["restart"]:
        out["opt_m"] = om
        if ov is not None:
            out["opt_v"] = ov
    if mode == "adamw":
        out["global_v"] = v
    return out
