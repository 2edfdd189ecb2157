"""The framework's work as its users call it, case by case, with inputs drawn from a seed.

A case is a dict of plain values; ``prepare`` makes what a program holds before
the call (observations on the GPU, the operator's factors, the handle, output
buffers), ``run`` makes one pass through the public API, ``work`` counts the
bytes and operations the pass cannot do without, and ``exact`` gives the same
outputs computed in 64 bits with torch and numpy alone.

The restoration problems follow the repository's workloads: piecewise-smooth
colour images (or translated smooth videos), a separable Gaussian blur with
zero boundary, a 3 x 3 channel mix, additive noise, GCV over eight values of
mu or a fixed mu, and a stop at the discrepancy level of the noise.
"""
import math
import random

import numpy as np
import torch

from paper_2603_00839_gb300 import api

MIX = [[0.8, 0.1, 0.1], [0.1, 0.8, 0.1], [0.1, 0.1, 0.8]]
GRID = [10.0 ** (-4.0 + 3.0 * i / 7.0) for i in range(8)]   # GCV candidates in [1e-4, 1e-1]
SAFETY = 1.5                                                # stop at this multiple of the noise level

_HANDLE = []


def _handle():
    # one handle for the whole program, as a user keeps it: plans and graphs live in it
    if not _HANDLE:
        _HANDLE.append(api.Handle(0))
    return _HANDLE[0]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # A small FP64 restoration with a fixed mu (the 64 x 64 x 3 configuration): every kernel is short, so
        # launches and dependent latencies are the whole time.
        {"name": "solve_f64_64", "kind": "solve", "dtype": "f64", "I1": 64, "I2": 64, "sigma": 1.5, "radius": 4,
         "mix": False, "nu": 1e-3, "m": 30, "s": 32, "lam": 1e-3, "stop": True},
        # The ordinary call: one 512 x 512 colour image in FP32, GCV, stopped at the noise level after a few steps.
        {"name": "solve_f32_512", "kind": "solve", "dtype": "f32", "I1": 512, "I2": 512, "sigma": 2.5, "radius": 7,
         "mix": True, "nu": 1e-3, "m": 50, "s": 128, "lam": -1.0, "stop": True},
        # A larger image run for its whole Krylov space (tol = 0, fixed mu): the basis outgrows the L2 cache.
        {"name": "solve_f32_1024", "kind": "solve", "dtype": "f32", "I1": 1024, "I2": 1024, "sigma": 2.5,
         "radius": 7, "mix": True, "nu": 2e-2, "m": 12, "s": 128, "lam": 1e-2, "stop": False},
        # An image of odd sides, as most photographs and crops are: nothing is a multiple of a tile or of 16 bytes.
        {"name": "solve_f32_ragged", "kind": "solve", "dtype": "f32", "I1": 333, "I2": 517, "sigma": 1.2,
         "radius": 4, "mix": False, "nu": 2e-2, "m": 20, "s": 128, "lam": 1e-2, "stop": False},
        # The serving form: many images of one camera at once, through the device work queue.
        {"name": "queue_512", "kind": "queue", "count": 48, "I1": 512, "I2": 512, "sigma": 2.5, "radius": 7,
         "nu": 2e-3, "m": 40, "s": 128, "slots": 8},
        # A mixed batch: images of all sizes, each with its own blur, noise and mu, as branches of one graph.
        {"name": "batch_ragged", "kind": "ragged", "count": 32, "lo": 64, "hi": 1024, "m": 30, "s": 128, "mix_seed": 1},
        # A colour video with a temporal blur, FP32 basis: the tensors are far larger than the L2 cache.
        {"name": "video_f32", "kind": "video", "I": 256, "frames": 64, "steps": 10},
        # The video's layers in BF16 storage, as the precision form runs them: the blurred video, and the sketch of one.
        {"name": "video_layers_bf16", "kind": "layers16", "I": 256, "frames": 64},
        # Sketched Golub-Kahan on the ordinary image, GCV.
        {"name": "gk_512", "kind": "gk", "I1": 512, "I2": 512, "sigma": 2.5, "radius": 7, "nu": 1e-2, "m": 10, "s": 128},
        # The layers alone on a large image: the blurred prediction of an iterate and its sketch.
        {"name": "apply_sketch_1024", "kind": "layers", "I1": 1024, "I2": 1024, "radius": 9, "s": 128},
        # The learned warm start at inference: one 512 x 512 image.
        {"name": "predict_512", "kind": "predict", "count": 1, "I1": 512, "I2": 512, "base": 32},
        # One training step of the warm start on a batch of 128 x 128 images (forward, loss, backward, Adam).
        {"name": "train_16x128", "kind": "train", "count": 16, "I1": 128, "I2": 128, "base": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the ranges above."""
    kind = rng.choice(["solve", "solve", "solve64", "queue", "ragged", "video", "layers16", "gk", "layers", "predict",
                       "train"])
    sigma = round(rng.uniform(0.5, 3.0), 3)
    radius = min(9, math.ceil(3 * sigma))
    nu = round(10 ** rng.uniform(-2.7, -1.7), 5)
    if kind == "solve":
        stop = rng.random() < 0.5
        return {"kind": "solve", "dtype": "f32", "I1": _log_int(rng, 64, 768), "I2": _log_int(rng, 64, 768),
                "sigma": sigma, "radius": radius, "mix": rng.random() < 0.5, "nu": nu if stop else 2e-2,
                "m": rng.randint(16, 40) if stop else rng.randint(8, 16), "s": rng.choice([64, 96, 128]),
                "lam": rng.choice([-1.0, 1e-3, 1e-2]) if stop else 1e-2, "stop": stop}
    if kind == "solve64":
        return {"kind": "solve", "dtype": "f64", "I1": _log_int(rng, 48, 160), "I2": _log_int(rng, 48, 160),
                "sigma": sigma, "radius": radius, "mix": rng.random() < 0.5, "nu": nu, "m": rng.randint(8, 30),
                "s": rng.choice([24, 32, 40]), "lam": rng.choice([-1.0, 1e-3]), "stop": rng.random() < 0.5}
    if kind == "queue":
        return {"kind": "queue", "count": rng.randint(8, 40), "I1": _log_int(rng, 128, 512),
                "I2": _log_int(rng, 128, 512), "sigma": sigma, "radius": radius, "nu": max(nu, 3e-3), "m": rng.randint(20, 40),
                "s": rng.choice([96, 128]), "slots": rng.choice([4, 8, 16])}
    if kind == "ragged":
        return {"kind": "ragged", "count": rng.randint(8, 32), "lo": 64, "hi": _log_int(rng, 256, 1000),
                "m": rng.randint(16, 30), "s": rng.choice([96, 128]), "mix_seed": rng.randint(2, 10 ** 6)}
    if kind == "video":
        return {"kind": "video", "I": 8 * rng.randint(10, 32), "frames": rng.randint(9, 64),
                "steps": rng.randint(4, 10)}
    if kind == "layers16":
        return {"kind": "layers16", "I": 8 * rng.randint(10, 32), "frames": rng.randint(9, 64)}
    if kind == "gk":
        return {"kind": "gk", "I1": _log_int(rng, 96, 640), "I2": _log_int(rng, 96, 640), "sigma": sigma,
                "radius": radius, "nu": nu, "m": rng.randint(5, 10), "s": rng.choice([64, 128])}
    if kind == "layers":
        return {"kind": "layers", "I1": _log_int(rng, 100, 1024), "I2": _log_int(rng, 100, 1024),
                "radius": rng.randint(2, 9), "s": rng.choice([64, 128])}
    if kind == "predict":
        return {"kind": "predict", "count": rng.randint(1, 4), "I1": 8 * rng.randint(12, 64), "I2": 8 * rng.randint(12, 64),
                "base": 32}
    return {"kind": "train", "count": rng.randint(4, 16), "I1": 8 * rng.randint(6, 16), "I2": 8 * rng.randint(6, 16),
            "base": 32}


# ---------------------------------------------------------------- inputs (torch only; mode 1 is the last axis)

def _gen(seed, stream):
    g = torch.Generator()
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFF)
    return g


def _noise(shape, seed, stream, dtype):
    g = torch.Generator(device=_device())
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFF)
    return torch.randn(shape, generator=g, device=_device(), dtype=dtype)


def _taps(sigma, radius):
    t = np.arange(-radius, radius + 1, dtype=np.float64)
    a = np.exp(-0.5 * (t / sigma) ** 2)
    return a / a.sum()


def _band(x, taps, axis):
    """y_i = sum_t taps[r + t] x_{i + t} along `axis`, zero outside."""
    r, n = (len(taps) - 1) // 2, x.shape[axis]
    y = torch.zeros_like(x)
    for t in range(-r, r + 1):
        w = n - abs(t)
        if w > 0:
            y.narrow(axis, max(0, -t), w).add_(x.narrow(axis, max(0, t), w), alpha=float(taps[r + t]))
    return y


def _images(count, I1, I2, seed, dtype):
    """(count, 3, I2, I1) piecewise-smooth colour images in [0, 1]: twenty rectangles in painter's order and a ramp."""
    g, dev = _gen(seed, 1), _device()
    x = torch.arange(I1, device=dev).view(1, 1, 1, I1)
    y = torch.arange(I2, device=dev).view(1, 1, I2, 1)
    img = torch.zeros((count, 3, I2, I1), dtype=dtype, device=dev)
    for _ in range(20):
        u = torch.rand((count, 4), generator=g, dtype=torch.float64)
        a = (torch.sort(u[:, :2], dim=1).values * I1).long().to(dev).view(count, 2, 1, 1, 1)
        b = (torch.sort(u[:, 2:], dim=1).values * I2).long().to(dev).view(count, 2, 1, 1, 1)
        val = torch.rand((count, 3, 1, 1), generator=g, dtype=torch.float64).to(dev, dtype)
        inside = (x >= a[:, 0]) & (x <= a[:, 1]) & (y >= b[:, 0]) & (y <= b[:, 1])
        img = torch.where(inside, val, img)
    return 0.5 * img + 0.25 * (x.to(dtype) / I1 + y.to(dtype) / I2)


def _mix(x, axis):
    """Channel mix by the symmetric matrix MIX along `axis`."""
    p = [x.select(axis, c) for c in range(3)]
    return torch.stack([MIX[o][0] * p[0] + MIX[o][1] * p[1] + MIX[o][2] * p[2] for o in range(3)], dim=axis)


def _observe(x, taps, mix, nu, seed, stream):
    """C = Phi(X) + N with ||N|| = nu ||Phi(X)|| per image (first axis)."""
    c = _band(_band(x, taps, 3), taps, 2)
    if mix:
        c = _mix(c, 1)
    e = _noise(c.shape, seed, stream, c.dtype)
    f = nu * c.flatten(1).norm(dim=1) / e.flatten(1).norm(dim=1)
    return c + e * f.view(-1, 1, 1, 1)


def _video(I, frames, seed):
    """(frames, 3, I, I): sixteen Gaussian bumps per channel on a wider canvas, moving one pixel a frame along mode 2."""
    g, dev = _gen(seed, 2), _device()
    x = torch.arange(I, device=dev, dtype=torch.float32).view(1, 1, I)
    y = torch.arange(I + frames, device=dev, dtype=torch.float32).view(1, I + frames, 1)
    canvas = torch.zeros((3, I + frames, I), device=dev)
    for _ in range(16):
        u = torch.rand((4, 3, 1, 1), generator=g).to(dev)
        w = I / 32.0 + u[2] * (I / 6.0 - I / 32.0)
        canvas += u[3] * torch.exp(-((x - u[0] * I) ** 2 + (y - u[1] * (I + frames)) ** 2) / (2 * w * w))
    lo, hi = canvas.amin(dim=(1, 2), keepdim=True), canvas.amax(dim=(1, 2), keepdim=True)
    canvas = (canvas - lo) / (hi - lo)
    return torch.stack([canvas[:, t:t + I, :] for t in range(frames)])


def _ragged(case):
    """The batch's problems: sides, blur, noise and mu of each."""
    r = random.Random(case["mix_seed"])
    out = []
    for _ in range(case["count"]):
        I1, I2 = r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"])
        sigma = r.uniform(0.5, 3.0)
        out.append({"I1": I1, "I2": I2, "sigma": sigma, "radius": math.ceil(3 * sigma), "nu": 10 ** r.uniform(-3.0, -2.3),
                    "lam": 10 ** r.uniform(-4.0, -1.0)})
    return out


def _tol(nu):
    return max(1e-3, SAFETY * nu)


def _operator(I1, I2, taps, mix):
    A = [api.banded(1, I1, taps), api.banded(2, I2, taps)]
    return A, [api.dense(3, np.array(MIX))] if mix else []


def _video_operator(case):
    A = [api.banded(1, case["I"], _taps(2.0, 6)), api.banded(2, case["I"], _taps(2.0, 6)),
         api.banded(4, case["frames"], np.full(5, 0.2))]
    return A, [api.dense(3, np.array(MIX))]


def _user(x):
    """The API's view of a (..., I2, I1) tensor: modes in order, mode 1 fastest."""
    return x.permute(*reversed(range(x.dim())))


def _problem(case, seed):
    """Observation(s) of a solve, queue, gk or video case, mode 1 on the last axis."""
    dt = torch.float64 if case.get("dtype") == "f64" else torch.float32
    if case["kind"] in ("video", "layers16"):
        x = _video(case["I"], case["frames"], seed)
        c = _mix(_band(_band(_band(x, _taps(2.0, 6), 3), _taps(2.0, 6), 2), np.full(5, 0.2), 0), 1)
        e = _noise(c.shape, seed, 3, c.dtype)
        return c + e * (5e-3 * c.norm() / e.norm())
    x = _images(case.get("count", 1), case["I1"], case["I2"], seed, dt)
    return _observe(x, _taps(case["sigma"], case["radius"]), case.get("mix", True), case["nu"], seed, 3)


def _sketch_dims(case, dims):
    return [min(case["s"], dims[0]), min(case["s"], dims[1]), 3]


def _video_sketch(case):
    s = max(1, (96 * case["I"]) // 256)
    return [s, s, 3, max(1, case["frames"] // 2)]


def _net_shapes(c):
    return [("e1", 3, c, 1), ("e2", c, 2 * c, 2), ("e3", 2 * c, 4 * c, 2), ("e4", 4 * c, 4 * c, 2),
            ("d3", 4 * c, 4 * c, 1), ("d2", 4 * c, 2 * c, 1), ("d1", 2 * c, c, 1), ("out", c, 3, 1)]


def _net(base, seed):
    """Parameters of a network that has been trained for a while: He-normal layers with small biases, and a small
    output layer and head (its correction of C is a few percent)."""
    rng = np.random.default_rng([int(seed), 5])
    P = {}
    for name, cin, cout, _ in _net_shapes(base):
        std = math.sqrt(2.0 / (9 * cin)) * (0.02 if name == "out" else 1.0)
        P[name + ".w"] = (rng.standard_normal((cout, 3, 3, cin)) * std).astype(np.float32)
        P[name + ".b"] = (rng.standard_normal(cout) * 0.02).astype(np.float32)
    P["lam.w"] = (rng.standard_normal(4 * base) * 0.05).astype(np.float32)
    P["lam.b"] = np.array([-5.0], dtype=np.float32)
    return P


def _net_inputs(case, seed):
    x = _images(case["count"], case["I1"], case["I2"], seed, torch.float32)
    c = _observe(x, _taps(1.5, 5), True, 5e-3, seed, 3)
    logmu = (torch.rand(case["count"], generator=_gen(seed, 6)) * 6.9 - 9.2).to(_device())
    return c.contiguous(), x.contiguous(), logmu


# ---------------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "gk"):
        h = _handle()
        c = _problem(case, seed)[0].contiguous()
        A, B = _operator(case["I1"], case["I2"], _taps(case["sigma"], case["radius"]), case.get("mix", True))
        return {"case": case, "h": h, "C": _user(c), "X": _user(torch.empty_like(c)), "A": A, "B": B,
                "seed": int(seed) & 0xFFFF}
    if kind == "video":
        c = _problem(case, seed).contiguous()
        A, B = _video_operator(case)
        return {"case": case, "h": _handle(), "C": _user(c), "X": _user(torch.empty_like(c)), "A": A, "B": B,
                "seed": int(seed) & 0xFFFF}
    if kind == "layers16":
        x = _problem(case, seed).to(torch.bfloat16).contiguous()
        A, B = _video_operator(case)
        return {"case": case, "h": _handle(), "X": _user(x), "Y": _user(torch.empty_like(x)),
                "SX": api.empty(_video_sketch(case)), "A": A, "B": B, "seed": int(seed) & 0xFFFF}
    if kind == "queue":
        c = _problem(case, seed).contiguous()
        A, B = _operator(case["I1"], case["I2"], _taps(case["sigma"], case["radius"]), True)
        out = torch.empty_like(c)
        probs = [dict(C=_user(c[i]), X=_user(out[i]), A=A, B=B, m=case["m"],
                      sketch_dims=_sketch_dims(case, (case["I1"], case["I2"])), seed=(int(seed) + i) & 0xFFFF, lam=-1.0,
                      tol=_tol(case["nu"])) for i in range(case["count"])]
        return {"case": case, "h": _handle(), "probs": probs}
    if kind == "ragged":
        probs = []
        for i, q in enumerate(_ragged(case)):
            taps = _taps(q["sigma"], q["radius"])
            c = _observe(_images(1, q["I1"], q["I2"], seed + 17 * i, torch.float32), taps, True, q["nu"], seed + 17 * i, 3)
            c = c[0].contiguous()
            A, B = _operator(q["I1"], q["I2"], taps, True)
            probs.append(dict(C=_user(c), X=_user(torch.empty_like(c)), A=A, B=B, m=case["m"],
                              sketch_dims=_sketch_dims(case, (q["I1"], q["I2"])), seed=(int(seed) + i) & 0xFFFF,
                              lam=q["lam"], tol=_tol(q["nu"])))
        return {"case": case, "h": _handle(), "probs": probs}
    if kind == "layers":
        x = _images(1, case["I1"], case["I2"], seed, torch.float32)[0].contiguous()
        A, B = _operator(case["I1"], case["I2"], _taps(case["radius"] / 3.0, case["radius"]), True)
        dims = (case["I1"], case["I2"], 3)
        sd = tuple(min(s, d) for s, d in zip(_sketch_dims(case, dims), dims))
        return {"case": case, "h": _handle(), "X": _user(x), "Y": api.empty(dims), "SY": api.empty(sd), "A": A, "B": B,
                "sd": sd, "seed": int(seed) & 0xFFFF}
    P = _net(case["base"], seed)
    net = api.WarmStart(case["base"], np.concatenate([v.ravel() for v in P.values()]))
    c, x, logmu = _net_inputs(case, seed)
    return {"case": case, "net": net, "C": c.view(-1), "Xs": x.view(-1), "logmu": logmu}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        X, info = state["h"].gmres_solve(
            state["C"], case["m"], _sketch_dims(case, (case["I1"], case["I2"])), state["seed"], case["lam"],
            A_factors=state["A"], B_factors=state["B"], X=state["X"], tol=_tol(case["nu"]) if case["stop"] else 0.0,
            mu_grid=GRID if case["lam"] < 0 else None)
        return {"X": X, "iters": info.iters}
    if kind == "gk":
        X, info = state["h"].gk_solve(
            state["C"], case["m"], _sketch_dims(case, (case["I1"], case["I2"])), state["seed"], -1.0,
            A_factors=state["A"], B_factors=state["B"], X=state["X"], mu_grid=GRID)
        return {"X": X, "iters": info.iters}
    if kind == "video":
        X, info = state["h"].gmres_solve(
            state["C"], case["steps"], _video_sketch(case), state["seed"], -1.0, A_factors=state["A"],
            B_factors=state["B"], X=state["X"], mu_grid=GRID)
        return {"X": X, "iters": info.iters}
    if kind == "queue":
        Xs, infos = state["h"].gmres_solve_batched(state["probs"], mu_grid=GRID, queue_slots=case["slots"])
        return {"X": Xs, "iters": np.array([r.iters for r in infos])}
    if kind == "ragged":
        Xs, infos = state["h"].gmres_solve_batched(state["probs"])
        return {"X": Xs, "iters": np.array([r.iters for r in infos])}
    if kind == "layers":
        Y = state["h"].operator_apply(state["X"], state["A"], state["B"], Y=state["Y"])
        SY = state["h"].sketch(Y, state["sd"], state["seed"], SX=state["SY"])
        return {"Y": Y, "SY": SY}
    if kind == "layers16":
        Y = state["h"].operator_apply(state["X"], state["A"], state["B"], Y=state["Y"])
        SX = state["h"].sketch(state["X"], _video_sketch(case), state["seed"], SX=state["SX"])
        return {"Y": Y, "SX": SX}
    if kind == "predict":
        X0, loglam = state["net"].predict(state["C"], case["I1"], case["I2"])
        return {"X0": X0, "loglam": loglam}
    loss = state["net"].train_step(state["C"], state["Xs"], state["logmu"], case["I1"], case["I2"], 1e-3)
    _, grads = state["net"].get()
    return {"loss": np.float32(loss), "grads": grads}


# ---------------------------------------------------------------- work

def _solve_work(n, d, b, m, ops, gk=False):
    # the observation is read, X written and, per step, the new basis tensor written and every one before it read
    # once; the operator and the sketch are counted in operations
    if gk:
        return {"bytes": b * (2 * n + m * 8 * n), "flops": m * 2 * ops}
    return {"bytes": b * (2 * n + sum((j + 2) * n + (j + 2) * d for j in range(m)) + (m + 1) * n), "flops": m * ops}


def work(case):
    kind = case["kind"]
    if kind in ("solve", "gk", "queue"):
        n = case["I1"] * case["I2"] * 3
        s1, s2 = min(case["s"], case["I1"]), min(case["s"], case["I2"])
        ops = 2 * n * (2 * (2 * case["radius"] + 1) + 3) + 2 * n * s1 + 2 * s1 * case["I2"] * 3 * s2
        steps = case["m"] if (kind == "gk" or not case.get("stop", True)) else min(case["m"], 8)
        w = _solve_work(n, s1 * s2 * 3, 8 if case.get("dtype") == "f64" else 4, steps, ops, kind == "gk")
        k = case.get("count", 1)
        return {"bytes": w["bytes"] * k, "flops": w["flops"] * k}
    if kind == "ragged":
        tot = {"bytes": 0, "flops": 0}
        for q in _ragged(case):
            n = q["I1"] * q["I2"] * 3
            s1, s2 = min(case["s"], q["I1"]), min(case["s"], q["I2"])
            ops = 2 * n * (2 * (2 * q["radius"] + 1) + 3) + 2 * n * s1 + 2 * s1 * q["I2"] * 3 * s2
            w = _solve_work(n, s1 * s2 * 3, 4, min(case["m"], 6), ops)
            tot = {"bytes": tot["bytes"] + w["bytes"], "flops": tot["flops"] + w["flops"]}
        return tot
    if kind == "video":
        n = case["I"] * case["I"] * 3 * case["frames"]
        s = _video_sketch(case)
        ops = 2 * n * (2 * 13 + 3 + 5) + 2 * n * s[0]
        return _solve_work(n, s[0] * s[1] * 3 * s[3], 4, case["steps"], ops)
    if kind == "layers16":
        n = case["I"] * case["I"] * 3 * case["frames"]
        s = _video_sketch(case)
        return {"bytes": 2 * 2 * n + 4 * s[0] * s[1] * 3 * s[3], "flops": 2 * n * (2 * 13 + 3 + 5) + 2 * n * s[0]}
    if kind == "layers":
        n, s = case["I1"] * case["I2"] * 3, case["s"]
        return {"bytes": 4 * (3 * n + 3 * s * s), "flops": 2 * n * (2 * (2 * case["radius"] + 1) + 3 + min(s, case["I1"]))}
    p, c = case["count"] * case["I1"] * case["I2"], case["base"]
    macs = p * 9 * (3 * c + c * 2 * c / 4 + 8 * c * c / 16 + 16 * c * c / 64 + 16 * c * c / 16 + 8 * c * c / 4 + 2 * c * c + 3 * c)
    acts = p * (2 * c + 3 * c / 2 + 12 * c / 16 + 4 * c / 64)
    if kind == "predict":
        return {"bytes": 4 * (6 * p + 2 * acts), "flops": 2 * macs}
    return {"bytes": 4 * (6 * p + 6 * acts), "flops": 6 * macs}


# ---------------------------------------------------------------- exact values (64 bits, torch and numpy)

def _thetas(dims, sdims, seed):
    """Rademacher matrices of the sketched modes (None: not sketched) from the Philox4x64-10 stream of `seed`."""
    sizes = [s * d if s < d else 0 for s, d in zip(sdims, dims)]
    words = np.random.Philox(key=int(seed)).random_raw((sum(sizes) + 63) // 64 + 1)
    bits = np.unpackbits(words.astype("<u8").view(np.uint8), bitorder="little")
    out, at = [], 0
    for s, d, k in zip(sdims, dims, sizes):
        if k == 0:
            out.append(None)
            continue
        sign = 1.0 - 2.0 * bits[at:at + k].astype(np.float64).reshape(s, d)
        out.append(torch.from_numpy(sign / math.sqrt(s)).to(_device()))
        at += k
    return out


def _mode(x, M, k):
    """Mode product of a tensor whose mode k is axis -(k + 1)."""
    ax = x.dim() - 1 - k
    return torch.movedim(torch.tensordot(M, x, dims=([1], [ax])), 0, ax)


def _sketch64(x, thetas):
    for k, t in enumerate(thetas):
        if t is not None:
            x = _mode(x, t, k)
    return x


def _choose(H, beta, lam):
    """The Tikhonov coefficients for mu = lam (0: least squares), or with mu chosen by GCV when lam < 0."""
    k = H.shape[1]
    b = np.zeros(k + 1)
    b[0] = beta

    def solve(mu):
        if mu == 0.0:
            return np.linalg.lstsq(H, b, rcond=None)[0]
        A = np.vstack([H, math.sqrt(mu) * np.eye(k)])
        return np.linalg.lstsq(A, np.concatenate([b, np.zeros(k)]), rcond=None)[0]

    if lam >= 0:
        return solve(lam)
    best = None
    for mu in GRID:
        y = solve(mu)
        T = np.eye(k + 1) - H @ np.linalg.solve(H.T @ H + mu * np.eye(k), H.T)
        v = float(np.sum((H @ y - b) ** 2)) / float(np.trace(T)) ** 2
        if best is None or v <= best[0]:
            best = (v, y)
    return best[1]


def _rho(H, beta):
    b = np.zeros(H.shape[0])
    b[0] = beta
    y = np.linalg.lstsq(H, b, rcond=None)[0]
    return float(np.linalg.norm(b - H @ y)) / beta


def _gmres64(C, phi, thetas, m, lam, tol):
    R = C.double()
    S = _sketch64(R, thetas)
    beta = float(S.norm())
    V, Q = [R / beta], [S.flatten() / beta]
    H = np.zeros((m + 1, m))
    k = m
    for j in range(m):
        W = phi(V[j])
        s = _sketch64(W, thetas).flatten()
        A = torch.stack(Q)
        h = A @ s
        s1 = s - A.T @ h
        h2 = A @ s1
        s1 = s1 - A.T @ h2
        h = h + h2
        hn = float(s1.norm())
        H[:j + 1, j] = h.cpu().numpy()
        H[j + 1, j] = hn
        for i in range(j + 1):
            W = W - h[i] * V[i]
        V.append(W / hn)
        Q.append(s1 / hn)
        if tol > 0 and _rho(H[:j + 2, :j + 1], beta) <= tol:
            k = j + 1
            break
    y = _choose(H[:k + 1, :k], beta, lam)
    return sum(float(y[i]) * V[i] for i in range(k)), k


def _gk64(C, phi, thetas, m):
    # the operator is symmetric (even taps, zero boundary, symmetric mix): its adjoint is itself
    norm = lambda x: float(_sketch64(x, thetas).norm())
    R = C.double()
    beta = norm(R)
    U = R / beta
    W = phi(U)
    alpha = norm(W)
    V, B = [W / alpha], np.zeros((m + 1, m))
    for j in range(m):
        B[j, j] = alpha
        W = phi(V[j]) - alpha * U
        b = norm(W)
        B[j + 1, j] = b
        U = W / b
        Z = phi(U) - b * V[j]
        alpha = norm(Z)
        V.append(Z / alpha)
    y = _choose(B, beta, -1.0)
    return sum(float(y[i]) * V[i] for i in range(m)), m


def _phi64(taps, mix):
    def phi(x):
        y = _band(_band(x, taps, x.dim() - 1), taps, x.dim() - 2)
        return _mix(y, x.dim() - 3) if mix else y
    return phi


def _net64(P, c, base):
    """The network's forward pass on (N, 3, I2, I1) images in 64 bits; returns X_0 and log lambda."""
    def conv(name, x, stride=1, relu=True):
        y = torch.nn.functional.conv2d(x, P[name + ".w"].permute(0, 3, 1, 2), P[name + ".b"], stride=stride, padding=1)
        return torch.relu(y) if relu else y
    up = lambda x: x.repeat_interleave(2, dim=2).repeat_interleave(2, dim=3)
    e1 = conv("e1", c)
    e2 = conv("e2", e1, 2)
    e3 = conv("e3", e2, 2)
    e4 = conv("e4", e3, 2)
    d3 = conv("d3", up(e4)) + e3
    d2 = conv("d2", up(d3)) + e2
    d1 = conv("d1", up(d2)) + e1
    return c + conv("out", d1, relu=False), e4.mean(dim=(2, 3)) @ P["lam.w"] + P["lam.b"]


def exact(case, seed):
    kind = case["kind"]
    seed = int(seed)
    with torch.no_grad():
        if kind in ("solve", "gk"):
            dims = (case["I1"], case["I2"], 3)
            th = _thetas(dims, _sketch_dims(case, dims), seed & 0xFFFF)
            phi = _phi64(_taps(case["sigma"], case["radius"]), case.get("mix", True))
            C = _problem(case, seed)[0]
            if kind == "gk":
                X, k = _gk64(C, phi, th, case["m"])
            else:
                X, k = _gmres64(C, phi, th, case["m"], case["lam"], _tol(case["nu"]) if case["stop"] else 0.0)
            return {"X": _user(X), "iters": k}
        if kind in ("video", "layers16"):
            taps = _taps(2.0, 6)
            dims = (case["I"], case["I"], 3, case["frames"])
            th = _thetas(dims, _video_sketch(case), seed & 0xFFFF)
            phi = lambda x: _mix(_band(_band(_band(x, taps, 3), taps, 2), np.full(5, 0.2), 0), 1)
            if kind == "layers16":
                x = _problem(case, seed).to(torch.bfloat16).double()
                return {"Y": _user(phi(x)), "SX": _user(_sketch64(x, th))}
            X, k = _gmres64(_problem(case, seed), phi, th, case["steps"], -1.0, 0.0)
            return {"X": _user(X), "iters": k}
        if kind in ("queue", "ragged"):   # the first few problems of the batch
            Xs = []
            for i in range(min(3, case["count"])):
                if kind == "queue":
                    q = dict(case, lam=-1.0)
                    C = _problem(case, seed)[i]
                else:
                    q = _ragged(case)[i]
                    x = _images(1, q["I1"], q["I2"], seed + 17 * i, torch.float32)
                    C = _observe(x, _taps(q["sigma"], q["radius"]), True, q["nu"], seed + 17 * i, 3)[0]
                dims = (q["I1"], q["I2"], 3)
                th = _thetas(dims, _sketch_dims(case, dims), (seed + i) & 0xFFFF)
                X, _ = _gmres64(C, _phi64(_taps(q["sigma"], q["radius"]), True), th, case["m"], q["lam"], _tol(q["nu"]))
                Xs.append(_user(X))
            return {"X": Xs + [None] * (case["count"] - len(Xs)), "iters": None}
        if kind == "layers":
            dims = (case["I1"], case["I2"], 3)
            x = _images(1, case["I1"], case["I2"], seed, torch.float32)[0].double()
            y = _phi64(_taps(case["radius"] / 3.0, case["radius"]), True)(x)
            th = _thetas(dims, [min(s, d) for s, d in zip(_sketch_dims(case, dims), dims)], seed & 0xFFFF)
            return {"Y": _user(y), "SY": _user(_sketch64(y, th))}
    P = {k: torch.from_numpy(v.astype(np.float64)).to(_device()) for k, v in _net(case["base"], seed).items()}
    c, x, logmu = (t.double() for t in _net_inputs(case, seed))
    if kind == "predict":
        with torch.no_grad():
            X0, ll = _net64(P, c, case["base"])
        return {"X0": X0.reshape(-1), "loglam": ll}
    for v in P.values():
        v.requires_grad_(True)
    X0, ll = _net64(P, c, case["base"])
    nrm = x.flatten(1).square().sum(dim=1)
    loss = (((X0 - x).flatten(1).square().sum(dim=1)) / nrm + (ll - logmu) ** 2).mean()
    g = torch.autograd.grad(loss, list(P.values()))
    return {"loss": float(loss), "grads": torch.cat([t.reshape(-1) for t in g]).cpu()}
