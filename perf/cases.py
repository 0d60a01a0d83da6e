"""The work a program has this framework do, as measured cases: worlds of robots stepped and read
back, training rows collected for the surrogate, its network trained and evaluated, and worlds
stepped by the surrogate.

Robots' results depend on the lanes that share a scene (the order of its sums), so a program that
wants to repeat its results fixes the launch shape, as these cases do; each takes the shape that
the autotuner settles on for its robots.  `uneven` runs untuned, in the shapes the library starts
with.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2411_05799_gb300 import npx, scenes

# The network of the surrogate of an 18-joint hexapod with six foot sensors.
N_IN, N_OUT, HIDDEN, LAYERS = 271, 247, 512, 4


def listed():
    return [
        # One robot between two joint updates of its controller: K steps, then the state and the
        # foot sensors come back.  Latency is all that counts.
        {"name": "control_1", "kind": "walk", "scenes": 1, "legs": 6, "steps": 80, "K": 80, "lanes": 32, "warps": 4,
         "friction": 0},
        # The ordinary batch: 4,096 hexapods on flat ground for one simulated second.
        {"name": "hexapods_4096", "kind": "walk", "scenes": 4096, "legs": 6, "steps": 1000, "K": 80, "lanes": 8,
         "warps": 7, "friction": 0},
        # The joint angles follow their targets at every step (K = 1), the costliest schedule.
        {"name": "every_step_4096", "kind": "walk", "scenes": 4096, "legs": 6, "steps": 100, "K": 1, "lanes": 16,
         "warps": 14, "friction": 0},
        # Evolution: 160 populations of 100 machine-code controllers, a slice of their evaluation.
        {"name": "evolution_16000", "kind": "evolve", "scenes": 16000, "steps": 400, "lanes": 8, "warps": 2},
        # Walkers on rough terrain, each on its own height map.
        {"name": "rough_4096", "kind": "rough", "scenes": 4096, "steps": 400, "cells": 64, "lanes": 16, "warps": 1},
        # Hexapods, quadrupeds and bipeds of 56 to about 1,000 points in one world.
        {"name": "uneven_8192", "kind": "uneven", "scenes": 8192, "steps": 200},
        # Robots that walk into one another, four to an arena.
        {"name": "arenas_1024x4", "kind": "arena", "arenas": 1024, "size": 4, "steps": 200, "lanes": 8, "warps": 1},
        # Training rows of the surrogate: eight windows of 25 steps of every robot.
        {"name": "collect_4096", "kind": "collect", "scenes": 4096, "stride": 25, "windows": 8, "lanes": 8,
         "warps": 7},
        # The statistics of one chunk of training rows.
        {"name": "moments_65536", "kind": "moments", "rows": 65536, "cols": N_IN},
        # Four minibatches of training, then the weights are taken out (a checkpoint).
        {"name": "train_8192", "kind": "train", "rows": 8192, "batches": 4, "n_in": N_IN, "hidden": HIDDEN,
         "layers": LAYERS, "n_out": N_OUT},
        # The network over every robot of a large world.
        {"name": "predict_65536", "kind": "predict", "rows": 65536, "n_in": N_IN, "hidden": HIDDEN, "layers": LAYERS,
         "n_out": N_OUT},
        # A world stepped by the surrogate for two joint-update periods; windows after which two or
        # more foot sensors would differ fall back to the plain step.
        {"name": "surrogate_16384", "kind": "surrogate", "scenes": 16384, "stride": 25, "steps": 160, "fallback": 1,
         "lanes": 8, "warps": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(robots, lanes):
    """The shape the autotuner tends to: one scene per warp for few robots, else the warps that spread
    the robots over 152 SMs once, or two-warp blocks where they do not fit at once."""
    if lanes == 32:
        return {"lanes": 32, "warps": 4}
    once = -(-robots * lanes // (152 * 32))
    return {"lanes": lanes, "warps": once if once * 32 // lanes <= 28 else 2}


def draw(rng):
    kind = rng.choice(["walk", "walk", "evolve", "rough", "uneven", "arena", "collect", "moments", "train", "predict",
                       "surrogate"])
    if kind == "walk":
        n, legs = _log(rng, 1, 8192), rng.choice([2, 4, 6, 6])
        K = rng.choice([1, 10, 80, 80, 80])
        steps = _log(rng, 20, 1000)
        steps = max(1, min(steps, (4096 * 1000 if K == 80 else 4096 * 100) // n))
        return {"kind": kind, "scenes": n, "legs": legs, "steps": steps, "K": K,
                **_shape(n, 32 if n < 256 else rng.choice([8, 8, 16])), "friction": rng.choice([0, 0, 0, 1, 2, 3])}
    if kind == "evolve":
        n = 100 * _log(rng, 1, 160)
        return {"kind": kind, "scenes": n, "steps": _log(rng, 80, 400), **_shape(n, 8)}
    if kind == "rough":
        return {"kind": kind, "scenes": _log(rng, 16, 4096), "steps": _log(rng, 50, 400),
                "cells": rng.choice([50, 64, 96]), "lanes": rng.choice([8, 16, 16]), "warps": 1}
    if kind == "uneven":
        return {"kind": kind, "scenes": _log(rng, 16, 8192), "steps": _log(rng, 20, 200)}
    if kind == "arena":
        size = rng.choice([2, 4])
        return {"kind": kind, "arenas": _log(rng, 1, 4096 // size), "size": size, "steps": _log(rng, 20, 200),
                "lanes": 8 if size == 4 else rng.choice([8, 16]), "warps": 1}
    if kind == "collect":
        n = _log(rng, 64, 4096)
        return {"kind": kind, "scenes": n, "stride": rng.randint(1, 39), "windows": rng.randint(1, 8), **_shape(n, 8)}
    if kind == "moments":
        return {"kind": kind, "rows": _log(rng, 100, 65536), "cols": rng.choice([N_IN, N_OUT, rng.randint(1, 300)])}
    if kind == "surrogate":
        n = _log(rng, 64, 16384)
        return {"kind": kind, "scenes": n, "stride": rng.choice([1, 16, 25, 26, 39]), "steps": rng.randint(80, 160),
                "fallback": rng.choice([-1, 0, 1]), **_shape(n, 8)}
    c = {"kind": kind, "n_in": rng.choice([N_IN, rng.randint(8, 300)]), "hidden": rng.choice([128, 256, 384, 512, 512]),
         "layers": rng.choice([1, 2, 4, 4]), "n_out": rng.choice([N_OUT, rng.randint(1, 300)])}
    if kind == "train":
        return {**c, "rows": 128 * _log(rng, 1, 64), "batches": rng.randint(1, 4)}
    return {**c, "rows": 128 * _log(rng, 1, 512)}


# ------------------------------------------------------------------------------------ inputs

def _world(batch, stream, case):
    shape = dict(lanes_per_scene=case["lanes"], warps_per_block=case["warps"]) if "lanes" in case else None
    return npx.World.from_batch(batch, stream=stream.cuda_stream, configure=shape)


def _reads(w):
    """Pinned arrays that the world's state is read into, pass after pass."""
    return {k: torch.from_numpy(a).pin_memory().numpy() for k, a in w.read_buffers().items()}


def _norms(w, S, stride, stream):
    """Standardisation of a world's training rows, from windows of the world itself."""
    nf, nt = npx.surrogate_dims(w)
    n = 3
    X, T = (torch.zeros(n * S, k, device="cuda") for k in (nf, nt))
    torch.cuda.synchronize()
    npx.surrogate_collect(w, n, X.data_ptr(), T.data_ptr(), stride=stride)
    stream.synchronize()

    def stat(a):
        mu, sd = a.double().mean(0), a.double().std(0, unbiased=False)
        return mu, torch.where(sd > 1e-6 * (mu.abs() + 1.0), sd, torch.ones_like(sd))

    (xm, xs), (tm, ts) = stat(X), stat(T)
    kept = [a.float().contiguous() for a in (xm, 1.0 / xs, tm, ts)]
    torch.cuda.synchronize()
    return kept, npx.SurrogateNorm(*[a.data_ptr() for a in kept])


def _weights(case, seed, last=1.0):
    """He-normal weights and small biases."""
    sizes = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
    rng = np.random.default_rng([seed, 1])
    Ws = [rng.standard_normal((o, i), dtype=np.float32) * np.float32(math.sqrt(2.0 / i))
          for i, o in zip(sizes[:-1], sizes[1:])]
    bs = [rng.standard_normal(o, dtype=np.float32) * np.float32(0.05) for o in sizes[1:]]
    Ws[-1] *= np.float32(last)
    bs[-1] *= np.float32(last)
    return Ws, bs


def _rows(case, seed):
    """Standardised features and targets (the targets only where a case trains)."""
    g = torch.Generator("cuda").manual_seed(seed)
    n = case["rows"] * case.get("batches", 1)
    x = torch.randn(n, case["n_in"], device="cuda", generator=g)
    if case["kind"] != "train":
        return x, None
    t = torch.randn(n, case["n_out"], device="cuda", generator=g)
    k = min(case["n_in"], case["n_out"])
    t[:, :k] = 0.5 * t[:, :k] + torch.tanh(x[:, :k])     # something that can be learned
    return x, t


def _moment_rows(case, seed):
    """Raw rows: columns of very different scale and offset, as the features have."""
    g = torch.Generator("cuda").manual_seed(seed)
    X = torch.randn(case["rows"], case["cols"], device="cuda", generator=g)
    k = torch.arange(case["cols"], device="cuda")
    return (X * 10.0 ** (k % 4 - 2) + (k % 7 - 3)).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    s = {"kind": kind, "case": case, "stream": stream}
    if kind in ("walk", "evolve", "rough", "uneven", "arena"):
        # a world whose robots already walk: past the drop onto their feet, not on a joint update
        if kind == "walk":
            batch = scenes.legged_batch(case["scenes"], case["legs"], seed_key=seed, K=case["K"])
        elif kind == "evolve":
            batch = scenes.hexapod_batch(case["scenes"], seed_key=seed)
        elif kind == "rough":
            batch = scenes.cpg_batch(case["scenes"], seed_key=seed, n_cells=case["cells"])
        elif kind == "uneven":
            # the same mix of robots; their friction and gaits come from the seed
            batch, rng = scenes.uneven_batch(case["scenes"]), np.random.default_rng(seed)
            gaits = rng.random((batch.n_joints, 4)) * [math.pi / 6, 1.5, 2 * math.pi, 0] + [0, 0.5, 0, 0]
            batch = batch.with_(mu=rng.uniform(0.3, 1.0, case["scenes"]).astype(np.float32),
                                act_params=gaits.astype(np.float32))
        else:
            batch = scenes.arena_batch(case["arenas"], case["size"], seed_key=seed)
        w = s["world"] = _world(batch, stream, case)
        if case.get("friction"):
            w.set_friction_model(case["friction"])
        if kind == "arena":
            w.set_arenas(case["size"], 0.01)
        if kind == "evolve":
            w.set_gp_programs(np.random.default_rng(seed).integers(0, 256, (case["scenes"], 32), dtype=np.uint8))
        w.step(201)
        w.sync()
        s["out"] = _reads(w)
    elif kind in ("collect", "surrogate"):
        w = s["world"] = _world(scenes.hexapod_batch(case["scenes"], seed_key=seed), stream, case)
        w.step(161)
        s["kept"], s["norm"] = _norms(w, case["scenes"], case["stride"], stream)
        nf, nt = npx.surrogate_dims(w)
        n = case["scenes"] * case.get("windows", 1)
        if kind == "collect":
            s["X"], s["T"] = torch.zeros(n, nf, device="cuda"), torch.zeros(n, nt, device="cuda")
        else:
            rows = (case["scenes"] + 127) // 128 * 128
            s["net"] = npx.MLP(nf, nt, n_hidden=HIDDEN, n_hidden_layers=LAYERS, max_batch=rows,
                               stream=stream.cuda_stream)
            # a network whose predictions stay near the mean change of a window, so that robots
            # move on plausibly without a training run here
            s["net"].set_params(*_weights({"n_in": nf, "hidden": HIDDEN, "layers": LAYERS, "n_out": nt}, seed, 0.02))
            npx.surrogate_set_fallback(w, case["fallback"])
            s["out"] = _reads(w)
    elif kind == "moments":
        s["X"] = _moment_rows(case, seed)
        s["sums"] = torch.zeros(2, case["cols"], dtype=torch.float64, device="cuda")
    else:
        s["x"], s["t"] = _rows(case, seed)
        s["net"] = npx.MLP(case["n_in"], case["n_out"], n_hidden=case["hidden"], n_hidden_layers=case["layers"],
                           max_batch=case["rows"], lr=1e-4, stream=stream.cuda_stream)
        s["net"].set_params(*_weights(case, seed))
        if kind == "train":
            s["loss"] = torch.zeros(case["batches"], device="cuda")
        else:
            s["y"] = torch.zeros(case["rows"], case["n_out"], device="cuda")
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------------------------ one pass

def run(state):
    s, case, kind = state, state["case"], state["kind"]
    if kind in ("walk", "evolve", "rough", "uneven", "arena"):
        s["world"].step(case["steps"])
        return s["world"].read(out=s["out"])
    if kind == "collect":
        npx.surrogate_collect(s["world"], case["windows"], s["X"].data_ptr(), s["T"].data_ptr(), s["norm"],
                              stride=case["stride"])
        return {"X": s["X"], "T": s["T"]}
    if kind == "surrogate":
        fell = npx.world_step_surrogate(s["world"], s["net"], s["norm"], case["steps"], stride=case["stride"])
        return {"fell_back": fell, **s["world"].read(out=s["out"])}
    if kind == "moments":
        with torch.cuda.stream(s["stream"]):
            s["sums"].zero_()
        npx.column_moments(s["X"].data_ptr(), case["rows"], case["cols"], s["sums"][0].data_ptr(),
                           s["sums"][1].data_ptr(), s["stream"].cuda_stream)
        return s["sums"]
    M = case["rows"]
    if kind == "predict":
        s["net"].forward(s["x"].data_ptr(), s["y"].data_ptr(), M)
        return s["y"]
    for b in range(case["batches"]):
        s["net"].backward(s["x"][b * M].data_ptr(), s["t"][b * M].data_ptr(), M, s["loss"][b:].data_ptr())
        s["net"].adam_step()
    Ws, bs = s["net"].get_params()
    return {"loss": s["loss"], "W": Ws, "b": bs}


# ------------------------------------------------------------------------------------ the floor

def work(case):
    """A step's operations as the paper writes it, in single precision: per point 18 (22 on a height
    map), per robot about 1,100 for the contacts, the friction fit and the integration, and about
    97 per point where the joints move.  Bytes: the robots once in, their state in and out."""
    kind = case["kind"]
    if kind == "moments":
        n = case["rows"] * case["cols"]
        return {"bytes": 4 * n + 16 * case["cols"], "flops": 3 * n}
    if kind in ("train", "predict"):
        sizes = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
        macs, n = sum(i * o for i, o in zip(sizes[:-1], sizes[1:])), case["rows"] * case.get("batches", 1)
        if kind == "predict":
            return {"bytes": 4 * n * (sizes[0] + sizes[-1]) + 4 * macs, "flops": 2 * n * macs}
        # the first layer needs no gradient of its input; weights, moments in and out per batch
        return {"bytes": 4 * n * (sizes[0] + sizes[-1]) + 24 * macs * case["batches"],
                "flops": 2 * n * (3 * macs - sizes[0] * sizes[1])}
    S = case.get("scenes") or case["arenas"] * case["size"]
    legs = case.get("legs", 6)
    points = 560 if kind == "uneven" else 64 + 48 * legs
    joints = 3 * legs
    per_robot = points * (17 + 2) + joints * 80 + 2 * 4 * 17
    steps = case["stride"] * case["windows"] if kind == "collect" else case["steps"]
    step = (22 if kind == "rough" else 18) * points + 1100
    flops = S * steps * (step + 97 * points / case.get("K", 80))
    nbytes = S * per_robot
    if kind == "collect":
        nbytes += 4 * S * case["windows"] * (N_IN + N_OUT)
    if kind == "surrogate":
        windows = (80 - 1) // case["stride"] * case["steps"] // 80
        macs = N_IN * HIDDEN + (LAYERS - 1) * HIDDEN * HIDDEN + HIDDEN * N_OUT
        flops = 2 * S * windows * macs + S * (case["steps"] - windows * case["stride"]) * step
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------ in 64 bits

def exact(case, seed):
    """The network's and the statistics' results in 64 bits.  Robots in contact have none: their
    paths part from any other rounding of theirs, contact by contact, within a window's steps."""
    kind = case["kind"]
    if kind == "moments":
        X = _moment_rows(case, seed).double()
        return torch.stack([X.sum(0), X.square().sum(0)])
    if kind not in ("train", "predict"):
        return None
    x, t = _rows(case, seed)
    Ws, bs = ([torch.from_numpy(a).cuda().double() for a in group] for group in _weights(case, seed))
    act = lambda z: torch.nn.functional.gelu(z, approximate="tanh")
    M = case["rows"]
    if kind == "predict":
        y = torch.empty(M, case["n_out"], dtype=torch.float64, device="cuda")
        for i in range(0, M, 8192):
            h = x[i:i + 8192].double()
            for W, b in zip(Ws[:-1], bs[:-1]):
                h = act(h @ W.T + b)
            y[i:i + 8192] = h @ Ws[-1].T + bs[-1]
        return y
    params = [p.requires_grad_() for pair in zip(Ws, bs) for p in pair]
    first, second = ([torch.zeros_like(p) for p in params] for _ in range(2))
    losses = []
    for k in range(case["batches"]):
        h = x[k * M:(k + 1) * M].double()
        for W, b in zip(Ws[:-1], bs[:-1]):
            h = act(h @ W.T + b)
        loss = (h @ Ws[-1].T + bs[-1] - t[k * M:(k + 1) * M].double()).square().sum() / M
        losses.append(loss.detach())
        grads = torch.autograd.grad(loss, params)
        with torch.no_grad():
            for p, g, m, v in zip(params, grads, first, second):
                m.mul_(0.9).add_(g, alpha=0.1)
                v.mul_(0.999).addcmul_(g, g, value=0.001)
                p -= 1e-4 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return {"loss": torch.stack(losses), "W": [W.detach() for W in Ws], "b": [b.detach() for b in bs]}
