"""The work a user has this library do, as a list of cases that can be timed and compared.

A case is one call sequence through `paper_2510_23498_b200.binding.Context`: either a training pass (forward solve, the caller's
loss head on the device, backward solve) or an inference pass (forward solve alone, which returns the stored trajectory).
`prepare` holds what a program keeps between passes: the context with its workspace, parameters, initial states, the grid and the
data of the loss head.
"""
import math

import numpy as np
import torch

from paper_2510_23498_b200 import binding

STAGES = {"euler": 1, "midpoint": 2, "heun": 2, "kutta3": 3, "rk4": 4, "rk38": 4}


def _case(name, kind, **kw):
    base = dict(name=name, kind=kind, train=True, batch=1, d=1, hidden=0, layers=0, act="softplus", side=0, channels=0, steps=1,
                solver="rk4", low="bf16", scaling="none", want_dt=False)
    base.update(kw)
    return base


def listed():
    return [
        # small calls: latency and launches count.  A toy flow map, fp16 with dynamic adjoint scaling
        _case("toy_mlp_train", "mlp", batch=512, d=2, hidden=32, layers=1, act="tanh", steps=10, low="f16", scaling="dynamic"),
        # the linear test equation: a long chain of small products
        _case("linear_train", "linear", batch=1024, d=64, steps=100),
        # the MLP block at full size: the benchmark's default workload
        _case("mlp_block_train", "mlp", batch=8192, d=256, hidden=1024, layers=2, steps=64),
        # a mid-sized MLP at sizes that are not tile multiples, fp16 with dynamic adjoint scaling
        _case("mlp_ragged_train", "mlp", batch=1000, d=72, hidden=200, layers=2, steps=16, low="f16", scaling="dynamic"),
        # serving the trained MLP block on a small, odd batch: forward only
        _case("mlp_block_infer", "mlp", train=False, batch=100, d=256, hidden=1024, layers=2, steps=32),
        # float32 mode: the accuracy reference a user trains against
        _case("mlp_f32_train", "mlp", batch=1024, d=64, hidden=256, layers=2, steps=16, low="f32"),
        # the convolutional classifier block at full size, fp16 with dynamic adjoint scaling
        _case("conv_block_train", "conv", batch=256, side=32, channels=64, act="relu", steps=8, low="f16", scaling="dynamic"),
        # the same block classifying an odd number of images
        _case("conv_block_infer", "conv", train=False, batch=37, side=32, channels=64, act="relu", steps=8, low="f16"),
        # the continuous normalizing flow with a trace estimate, image-sized state
        _case("cnf_train", "cnf", batch=2048, d=784, hidden=2048, layers=2, steps=8),
        # the same flow on tabular data: an odd feature count
        _case("cnf_tabular_train", "cnf", batch=512, d=63, hidden=1024, layers=2, steps=16),
        # two-dimensional flow with the exact trace: many small steps, fp16 with dynamic adjoint scaling
        _case("hyper_cnf_train", "cnf_hyper", batch=1024, d=2, hidden=32, channels=128, steps=128, low="f16", scaling="dynamic"),
        # the parabolic convolutional block with 512 channels
        _case("parabolic_train", "parabolic", batch=16, side=32, channels=512, act="relu", steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """Mostly multiples of 8, as people choose them, now and then an odd width."""
    w = _log_int(rng, lo, hi)
    return w if rng.random() < 0.2 else max(8, (w + 4) // 8 * 8)


def draw(rng):
    kind = rng.choice(["toy", "linear", "mlp", "mlp", "f32", "conv", "cnf", "cnf", "cnf_hyper", "parabolic"])
    low, scaling = rng.choice([("bf16", "none"), ("bf16", "none_safe"), ("f16", "dynamic")])
    solver = rng.choice(["rk4", "rk4", "rk4", "heun", "euler"])
    train = rng.random() < 0.75
    if kind == "toy":
        c = _case("", "mlp", batch=_log_int(rng, 16, 1024), d=rng.randint(2, 4), hidden=rng.randint(8, 64), layers=1,
                  act=rng.choice(["tanh", "softplus"]), steps=_log_int(rng, 4, 40), want_dt=train and rng.random() < 0.2)
    elif kind == "linear":
        c = _case("", "linear", batch=_log_int(rng, 64, 4096), d=_width(rng, 16, 128), steps=_log_int(rng, 20, 100))
    elif kind in ("mlp", "f32"):
        c = _case("", "mlp", batch=_log_int(rng, 64, 8192 if kind == "mlp" else 2048), d=_width(rng, 16, 256),
                  hidden=_width(rng, 64, 1024 if kind == "mlp" else 512), layers=rng.randint(1, 2),
                  act=rng.choice(["softplus", "tanh", "relu"]), steps=_log_int(rng, 4, 64), want_dt=train and rng.random() < 0.15)
        if kind == "f32":
            low, scaling = "f32", "none"
    elif kind == "conv":
        c = _case("", "conv", batch=_log_int(rng, 4, 256), side=rng.choice([8, 16, 32]), channels=rng.choice([16, 64, 64, 64]),
                  act=rng.choice(["relu", "softplus"]), steps=_log_int(rng, 2, 8))
    elif kind == "cnf":
        c = _case("", "cnf", batch=_log_int(rng, 64, 2048), d=_width(rng, 16, 784), hidden=_width(rng, 64, 2048), layers=rng.randint(1, 2),
                  steps=_log_int(rng, 4, 16))
    elif kind == "cnf_hyper":
        c = _case("", "cnf_hyper", batch=_log_int(rng, 64, 4096), d=2, hidden=rng.choice([16, 32, 64]), channels=rng.choice([32, 64, 128, 256]),
                  steps=_log_int(rng, 8, 128))
    else:
        c = _case("", "parabolic", batch=_log_int(rng, 2, 16), side=rng.choice([16, 32]), channels=rng.choice([64, 128, 256, 512]),
                  act="relu", steps=_log_int(rng, 2, 6))
    c.update(low=low, scaling=scaling, solver=solver, train=train)
    # no drawn case is more work than the largest listed one; shapes that run on the CUDA cores are kept smaller
    odd = low == "f32" or (c["channels"] % 64 if kind in ("conv", "parabolic") else c["d"] % 8 or c["hidden"] % 8)
    most = 2e11 if odd else 1e13
    while _flops(c) > most and (c["batch"] > 2 or c["steps"] > 1):
        if c["batch"] > 16 or c["steps"] == 1:
            c["batch"] = max(2, c["batch"] * 2 // 3)
        else:
            c["steps"] = max(1, c["steps"] * 2 // 3)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ sizes
def _widths(c):
    return [c["d"]] + [c["hidden"]] * c["layers"] + [c["d"]]


def _state(c):
    """stored state width d of one sample, and the width D of the solved state (the flows carry a log-density)"""
    d = c["side"] * c["side"] * c["channels"] if c["kind"] in ("conv", "parabolic") else c["d"]
    return d, d + 1 if c["kind"] in ("cnf", "cnf_hyper") else d


def _params(c):
    k, C = c["kind"], c["channels"]
    if k == "linear":
        return c["d"] * c["d"]
    if k in ("mlp", "cnf"):
        w = _widths(c)
        return sum(w[i + 1] * (w[i] + (1 if i == 0 else 0)) + w[i + 1] for i in range(len(w) - 1))
    if k == "conv":
        return 9 * C * (C + 1) + C + 9 * C * C + C
    if k == "parabolic":
        return c["steps"] * (9 * C * C + C)
    h, m = c["hidden"], C * (2 * c["d"] + 1)
    return 3 * h + h * h + m * h + m


def _flops(c):
    """Contractions of one pass: one evaluation per stage forward; backward again one, and twice that for the two products of Eq. (vjp)."""
    k, C = c["kind"], c["channels"]
    if k == "linear":
        macs = c["d"] * c["d"]
    elif k in ("mlp", "cnf"):
        w = _widths(c)
        macs = sum(a * b for a, b in zip(w[:-1], w[1:])) * (2 if k == "cnf" else 1)      # the flow: a tangent row beside every state
    elif k in ("conv", "parabolic"):
        macs = 2 * 9 * C * C * c["side"] * c["side"]
    else:
        macs = C * (2 * c["d"] + 2)
    return 2.0 * macs * c["batch"] * c["steps"] * STAGES[c["solver"]] * (4 if c["train"] else 1)


def work(case):
    d, D = _state(case)
    B, n, es = case["batch"], case["steps"], 4 if case["low"] == "f32" else 2
    p = _params(case)
    traj = (n + 1) * B * d * es
    nbytes = 4 * p + 4 * B * d + 4 * B * D + traj                  # parameters and y0 in, y_N and the trajectory out
    if case["kind"] == "cnf":
        nbytes += B * d
    if case["train"]:
        nbytes += traj + 4 * p + 4 * B * D * 2 + 4 * p             # the trajectory and parameters back, dL/dy_N in, both gradients out
    return {"bytes": nbytes, "flops": _flops(case)}


def tolerance(case):
    # Measured between two runs of the same network with its hidden units, channels or weight sets in another order, so that every sum
    # runs in another order: float32 1.8e-7; 16-bit layer outputs and cotangents that then round to a neighbour 1.3e-4 (fp16) and
    # 9e-4 (bf16).  Through a ReLU the units nearest their kink flip their derivative as well: 1.5e-4, 5e-3 (fp16), 1.5e-2 (bf16,
    # through instance normalisation).
    if case["act"] == "relu":
        return {"f32": {"rel": 1e-3, "max": 0.12}, "f16": {"rel": 2e-2, "max": 0.7}, "bf16": {"rel": 3e-2, "max": 0.9}}[case["low"]]
    return {"f32": {"rel": 1e-5, "max": 1e-4}, "f16": {"rel": 1e-3, "max": 1e-2}, "bf16": {"rel": 4e-3, "max": 5e-2}}[case["low"]]


# ------------------------------------------------------------------------------------------------ inputs
def _velocity(c):
    k = c["kind"]
    d, _ = _state(c)
    if k == "linear":
        return dict(kind="linear", d=d, widths=[d, d], act="none", append_time=False, bias=False)
    if k in ("mlp", "cnf"):
        return dict(kind=k, d=d, widths=_widths(c), act="softplus" if k == "cnf" else c["act"], append_time=True, bias=True)
    if k == "conv":
        return dict(kind="conv", d=d, H=c["side"], W=c["side"], C=c["channels"], act=c["act"], append_time=True)
    if k == "parabolic":
        return dict(kind="parabolic", d=d, H=c["side"], W=c["side"], C=c["channels"], n_intervals=c["steps"], norm=True, act="relu")
    return dict(kind="cnf_hyper", d=d, hidden=c["hidden"], w=c["channels"])


def _theta(c, randn):
    """Flat parameters in the library's layout: weights N(0, 1 / fan_in) (He for the convolutions), small biases."""
    k, C = c["kind"], c["channels"]
    parts = []
    if k == "linear":      # A = -Q diag(lam) Q^T, lam log-uniform in [0.1, 10]
        q, r = torch.linalg.qr(randn(c["d"], c["d"]).double())
        q = q * torch.sign(torch.diagonal(r))[None, :]
        lam = 10.0 ** (torch.erf(randn(c["d"]).double() / math.sqrt(2.0)))
        return (-(q * lam[None, :]) @ q.T).float().reshape(-1).contiguous()
    if k in ("mlp", "cnf"):
        w = _widths(c)
        for i in range(len(w) - 1):
            fan = w[i] + (1 if i == 0 else 0)
            parts += [randn(w[i + 1], fan) / math.sqrt(fan), 0.02 * randn(w[i + 1])]
    elif k == "conv":
        parts = [randn(C, 3, 3, C + 1) * math.sqrt(2.0 / (9 * (C + 1))), 0.02 * randn(C), randn(C, 3, 3, C) * math.sqrt(2.0 / (9 * C)), 0.02 * randn(C)]
    elif k == "parabolic":
        for _ in range(c["steps"]):
            parts += [randn(C, 3, 3, C) * math.sqrt(1.0 / (27 * C)), 0.1 * randn(C)]
    else:
        h, m = c["hidden"], C * (2 * c["d"] + 1)
        parts = [randn(h, 1), 0.02 * randn(h), randn(h, h) / math.sqrt(h), 0.02 * randn(h), randn(m, h) / math.sqrt(h), 0.02 * randn(m)]
    return torch.cat([x.reshape(-1) for x in parts]).contiguous()


def prepare(case, seed):
    c = case
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))

    def randn(*shape):
        return torch.randn(shape, generator=gen, device=dev, dtype=torch.float32)

    d, D = _state(c)
    B = c["batch"]
    # k_max: the pooled classification loss gives every pixel of an image the same cotangent, so that the first step's weight
    # gradient adds up coherently and the scale is halved more than ten times before it fits fp16
    ctx = binding.Context(_velocity(c), B, c["steps"], low=c["low"], scaling=c["scaling"], k_max=40, time_gradient=c["want_dt"])
    s = {"case": c, "ctx": ctx, "theta": _theta(c, randn), "tgrid": np.linspace(0.0, 1.0, c["steps"] + 1).astype(np.float32), "probe": None}
    if c["kind"] == "cnf_hyper":      # points on two noisy rings
        ang = 2.0 * math.pi * torch.rand((B,), generator=gen, device=dev)
        rad = 1.0 + 1.5 * (torch.rand((B,), generator=gen, device=dev) > 0.5) + 0.1 * randn(B)
        s["y0"] = torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], dim=1).float().contiguous()
    else:
        s["y0"] = randn(B, d)
    if c["kind"] == "cnf":
        s["probe"] = torch.where(randn(B, d) > 0, 1, -1).to(torch.int8)
    if c["train"]:
        if c["kind"] == "conv":
            s["head"] = randn(10, c["channels"]) / math.sqrt(c["channels"])
            s["labels"] = torch.randint(0, 10, (B,), generator=gen, device=dev)
        elif c["kind"] not in ("cnf", "cnf_hyper"):
            s["target"] = randn(B, d)
    return s


def _loss_head(s, yT):
    """The caller's loss and dL/dy_N: mean-squared error, pooled linear classifier, or the likelihood under a standard normal."""
    c = s["case"]
    B = c["batch"]
    if c["kind"] in ("cnf", "cnf_hyper"):
        z, ell = yT[:, :-1], yT[:, -1]
        loss = (0.5 * (z * z).sum(dim=1) + ell).mean()
        dl = yT / B
        dl[:, -1] = 1.0 / B
        return loss, dl
    if c["kind"] == "conv":
        feat = yT.view(B, c["side"] * c["side"], c["channels"]).mean(dim=1)
        logp = torch.log_softmax(feat @ s["head"].T, dim=1)
        loss = torch.nn.functional.nll_loss(logp, s["labels"])
        dlog = logp.exp() - torch.nn.functional.one_hot(s["labels"], 10)
        dfeat = (dlog / (B * c["side"] * c["side"])) @ s["head"]
        return loss, dfeat[:, None, :].expand(B, c["side"] * c["side"], c["channels"]).reshape(B, -1)
    r = yT - s["target"]
    return (r * r).mean(), r * (2.0 / r.numel())


def run(s):
    c, ctx = s["case"], s["ctx"]
    traj, yT = ctx.forward(s["theta"], s["y0"], s["tgrid"], c["solver"], s["probe"])
    if not c["train"]:
        return {"traj": traj, "yT": yT}
    loss, dl = _loss_head(s, yT)
    dy0, dtheta, log, status = ctx.backward(dl, want_dt=c["want_dt"])
    out = {"yT": yT, "loss": loss, "dy0": dy0, "dtheta": dtheta, "status": status}
    if c["want_dt"]:
        out["dt"] = log["dL_dt"]
    return out
