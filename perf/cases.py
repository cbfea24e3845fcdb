"""The work a user has this engine do, as cases that can be timed and compared.

Kinds of case:

  job       one lattice from the flat start through `mcs` sweeps with the exact
            W^2 at log-spaced times (Lattice.reset / run / roughness), the
            lattice kept in a caller-owned device buffer: the paper's single
            simulation, over sizes, rates and decompositions;
  ensemble  realisations of unequal L, p and run length in one persistent
            launch, and their W^2 curves (Batch.run / w2);
  gradient  loss and gradient of the surrogate's network over points of W^2
            curves, the step its training repeats (MLP.loss_grad);
  predict   its predictions along curves (MLP.predict);
  surface   a surface imported from packed slopes, its W^2, its heights and
            its slopes exported again (Lattice.set_slopes / roughness /
            heights / slopes): analysis of stored or foreign surfaces.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1204_5072_gb300 import Batch, Lattice
from paper_1204_5072_gb300 import surrogate

MLP_WIDTH = 128
MLP_PARAMS = 33793


def listed():
    return [
        # The validation run: small lattice, every sweep a latency-bound step.
        {"name": "job_L256_p1", "kind": "job", "L": 256, "p": 1.0, "q": 0.0, "mcs": 1000, "samples": 16,
         "decomposition": 0, "cell": 4, "tile_y": 128},
        # A curve W^2(t) of a mid-size lattice at general rates, as sampled for growth exponents.
        {"name": "job_L1024_p095", "kind": "job", "L": 1024, "p": 0.95, "q": 0.05, "mcs": 300, "samples": 24,
         "decomposition": 0, "cell": 4, "tile_y": 128},
        # The paper's single-GPU size range, at its benchmark rates and at general ones.
        {"name": "job_L4096_p1", "kind": "job", "L": 4096, "p": 1.0, "q": 0.0, "mcs": 200, "samples": 12,
         "decomposition": 0, "cell": 4, "tile_y": 128},
        {"name": "job_L4096_p095", "kind": "job", "L": 4096, "p": 0.95, "q": 0.05, "mcs": 101, "samples": 8,
         "decomposition": 0, "cell": 4, "tile_y": 128},
        # A large lattice with real deposition and evaporation.
        {"name": "job_L16384_p06_q03", "kind": "job", "L": 16384, "p": 0.6, "q": 0.3, "mcs": 40, "samples": 6,
         "decomposition": 0, "cell": 4, "tile_y": 128},
        # The headline lattice (4.3e9 sites), a short stretch of the 2000-sweep job.
        {"name": "job_L65536_p1", "kind": "job", "L": 65536, "p": 1.0, "q": 0.0, "mcs": 48, "samples": 6,
         "decomposition": 0, "cell": 4, "tile_y": 128},
        # Random-sequential reference the decompositions are checked against.
        {"name": "rsu_L1024_p095", "kind": "job", "L": 1024, "p": 0.95, "q": 0.05, "mcs": 8, "samples": 4,
         "decomposition": 4, "cell": 4, "tile_y": 128},
        # Device-layer double tiling (four tile sets, no dead border).
        {"name": "tilesets_L2048_p1", "kind": "job", "L": 2048, "p": 1.0, "q": 0.0, "mcs": 64, "samples": 8,
         "decomposition": 1, "cell": 4, "tile_y": 128},
        # A scaled-down batched workload: L = 256..8192, p in [0.5, 1], q = 1 - p.
        {"name": "ensemble_40", "kind": "ensemble", "n": 40, "mix": 1, "cap": 400, "samples": 32},
        # A minibatch's forward and backward pass, the unit of the surrogate's training.
        {"name": "gradient_128", "kind": "gradient", "n": 128},
        # One predicted curve, as the planner asks for per realisation.
        {"name": "predict_251", "kind": "predict", "n": 251},
        # Stored surface in, width, heights and slopes out.
        {"name": "surface_L2048", "kind": "surface", "L": 2048},
    ]


def draw(rng):
    kind = rng.choice(["job", "job", "job", "variant", "ensemble", "gradient", "predict", "surface"])
    if kind in ("job", "variant"):
        variant = kind == "variant"
        decomposition = rng.choice([1, 2, 3, 4]) if variant else 0
        log2L = rng.randint(8, 11) if variant else rng.randint(7, 15)
        L = 1 << log2L
        p, q = rng.choice([(1.0, 0.0), (round(rng.uniform(0.5, 0.999), 3), None),
                           (round(rng.uniform(0.1, 0.9), 3), round(rng.uniform(0.05, 0.9), 3))])
        q = round(1.0 - p, 3) if q is None else q
        budget = 2e10 if not variant else {1: 4e8, 2: 1e8, 3: 1e8, 4: 1e7}[decomposition]
        most = max(2, min(1000, int(budget / (L * L))))
        mcs = int(round(math.exp(rng.uniform(math.log(max(2.0, most / 8)), math.log(most)))))
        cell = 2 if not variant and rng.random() < 0.1 else 4
        tall = not variant and cell == 4 and L >= 256 and rng.random() < 0.2
        return {"kind": "job", "L": L, "p": p, "q": q, "mcs": mcs, "samples": rng.randint(2, 20),
                "decomposition": decomposition, "cell": cell, "tile_y": 256 if tall else 128}
    if kind == "ensemble":
        n = int(round(math.exp(rng.uniform(math.log(2), math.log(32)))))
        return {"kind": "ensemble", "n": n, "mix": rng.randint(2, 10 ** 6), "cap": rng.randint(60, 250),
                "samples": rng.randint(4, 48)}
    if kind == "gradient":
        return {"kind": "gradient", "n": int(round(math.exp(rng.uniform(math.log(16.0), math.log(5e4)))))}
    if kind == "predict":
        return {"kind": "predict", "n": int(round(math.exp(rng.uniform(0.0, math.log(3e5)))))}
    return {"kind": "surface", "L": 1 << rng.randint(7, 12), "h00": rng.randint(-9, 9)}


# --------------------------------------------------------------------------- #
def _times(T, n):
    """Log-spaced W^2 times 0 = t_0 < ... < t_m = T."""
    ts = {0, T}
    for k in range(n):
        ts.add(min(T, int(math.ceil(10 ** (k * math.log10(T) / max(1, n - 1)) - 1e-9))))
    return sorted(ts)


def _mix(case):
    """(L, run length) of an ensemble's realisations: L log-uniform in
    256..8192, run length 4 L^1.6 against a cap of 10^5, scaled to `cap`."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["n"]):
        L = 1 << r.randint(8, 13)
        out.append((L, max(1, math.ceil(min(4 * L ** 1.6, 1e5) * case["cap"] / 1e5))))
    return out


def _curve_points(n, rng):
    """Scaled features of n points (L, t, p, q = 1 - p) and targets following a growth law."""
    L = 2.0 ** rng.integers(8, 14, n)
    t = np.round(10 ** rng.uniform(0, 5, n))
    p = rng.uniform(0.5, 1.0, n)
    x = np.stack([(np.log2(L) - 10.0) / 2.0, (np.log(t) - 6.0) / 3.0, (p - 0.75) / 0.2, (0.75 - p) / 0.2], axis=-1)
    beta = 0.06 + 0.18 * (2 * p - 1)
    y = np.log(0.2 + 0.15 * t ** (2 * beta)) + 0.05 * rng.standard_normal(n)
    return x.astype(np.float32), y.astype(np.float32)


def _params(seed):
    """He-uniform weights and zero biases, the network's usual start."""
    rng, W, parts = np.random.default_rng(seed), MLP_WIDTH, []
    for fan_in in (4, W, W):
        a = math.sqrt(6.0 / fan_in)
        parts += [rng.uniform(-a, a, W * fan_in), np.zeros(W)]
    parts += [rng.uniform(-math.sqrt(3.0 / W), math.sqrt(3.0 / W), W), np.zeros(1)]
    return np.concatenate(parts).astype(np.float32)


def _walk(L, rng):
    s = np.repeat(np.array([0, 1], np.uint32), L // 2)
    rng.shuffle(s)
    return s


def _surface(case, seed):
    """A valid surface h(i,j) = f(i) + g(j): its +-1 steps (as 0/1) and its packed slopes."""
    L = case["L"]
    rng = np.random.default_rng(seed)
    sx, sy = _walk(L, rng), _walk(L, rng)
    row = (sx.reshape(-1, 16) << (2 * np.arange(16, dtype=np.uint32))).sum(axis=1, dtype=np.uint32)
    col = np.where(sy == 1, np.uint32(0xAAAAAAAA), np.uint32(0))
    return sx, sy, np.ascontiguousarray(row[None, :] | col[:, None]).reshape(-1)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "job":
        L = case["L"]
        buf = torch.empty(Lattice.device_bytes(L), dtype=torch.uint8, device="cuda")
        lat = Lattice(L, case["p"], case["q"], seed=seed, device_buffer=buf, tile_y=case["tile_y"],
                      decomposition=case["decomposition"], cell=case["cell"])
        return {"kind": kind, "lat": lat, "times": _times(case["mcs"], case["samples"]),
                "sites": buf[:L * L // 8].view(torch.int32)}
    if kind == "ensemble":
        rng = np.random.default_rng(seed)
        p = rng.uniform(0.5, 1.0, case["n"])
        specs = [(L, float(p[k]), float(1.0 - p[k]), seed, k, n) for k, (L, n) in enumerate(_mix(case))]
        return {"kind": kind, "batch": Batch(specs, n_samples=case["samples"], autotune=True, tile_y=128)}
    if kind == "gradient":
        x, y = _curve_points(case["n"], np.random.default_rng(seed))
        return {"kind": kind, "x": x, "y": y, "mlp": surrogate.MLP(_params(seed))}
    if kind == "predict":
        x, _ = _curve_points(case["n"], np.random.default_rng(seed))
        return {"kind": kind, "x": x, "mlp": surrogate.MLP(_params(seed))}
    words = _surface(case, seed)[2]
    return {"kind": kind, "lat": Lattice(case["L"], seed=seed), "words": words, "h00": case.get("h00", 0)}


def run(state):
    kind = state["kind"]
    if kind == "job":
        lat = state["lat"].reset()
        done, curve = 0, []
        for t in state["times"]:
            if t > done:
                lat.run(t - done)
                done = t
            curve.append(lat.roughness())
        return {"w2": np.array([r["w2"] for r in curve]), "S1": np.array([r["S1"] for r in curve], np.int64),
                "S2": np.array([r["S2"] for r in curve], np.int64), "h00": np.array([r["h00"] for r in curve], np.int64),
                "sites": state["sites"]}
    if kind == "ensemble":
        b = state["batch"].run()
        return {"w2": b.w2(), "times": b.times().astype(np.int64)}
    if kind == "gradient":
        loss, grad = state["mlp"].loss_grad(state["x"], state["y"])
        return {"loss": np.array([loss], np.float32), "grad": grad}
    if kind == "predict":
        return {"y": state["mlp"].predict(state["x"])}
    lat = state["lat"].set_slopes(state["words"], h00=state["h00"], t=0)
    r = lat.roughness()
    return {"w2": np.array([r["w2"]]), "S1": r["S1"], "S2": r["S2"], "heights": lat.heights(absolute=True),
            "slopes": lat.slopes().view(np.int32)}


def work(case):
    kind = case["kind"]
    if kind == "job":          # one bit read and one written per site and sweep, one read per W^2 sample
        sites = case["L"] ** 2
        return {"bytes": sites / 4 * case["mcs"] + sites / 8 * len(_times(case["mcs"], case["samples"])), "flops": 0}
    if kind == "ensemble":
        return {"bytes": sum(L * L / 4 * n for L, n in _mix(case)), "flops": 0}
    layer = 2 * MLP_WIDTH * MLP_WIDTH
    forward = 2 * layer + 2 * MLP_WIDTH * 5
    if kind == "gradient":     # samples, weights and gradient once; forward and backward
        return {"bytes": 20.0 * case["n"] + 6 * MLP_PARAMS, "flops": 3.0 * forward * case["n"]}
    if kind == "predict":
        return {"bytes": 20.0 * case["n"] + 2 * MLP_PARAMS, "flops": float(forward) * case["n"]}
    sites = case["L"] ** 2     # slopes in and out at 2 bits, heights out at 8 bytes
    return {"bytes": sites * (0.25 + 0.25 + 8.0), "flops": 0}


# --------------------------------------------------------------------------- #
def _bf16(a):
    return torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).to(torch.float64)


def _split(theta):
    W, out, k = MLP_WIDTH, [], 0
    for shape in ((W, 4), (W,), (W, W), (W,), (W, W), (W,), (W,), (1,)):
        n = int(np.prod(shape))
        out.append(theta[k:k + n].reshape(shape))
        k += n
    return out


def _forward(theta, x):
    W1, b1, W2, b2, W3, b3, w4, b4 = _split(theta)
    gelu = torch.nn.functional.gelu
    return gelu(gelu(gelu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3) @ w4 + b4


def exact(case, seed):
    """The network's results in 64 bits at its bfloat16 weights, and the width
    of a separable surface; lattice trajectories are whole numbers."""
    kind = case["kind"]
    if kind == "predict":
        x, _ = _curve_points(case["n"], np.random.default_rng(seed))
        y = _forward(_bf16(_params(seed)), torch.from_numpy(x).double())
        return {"y": y.numpy()}
    if kind == "gradient":
        x, y = _curve_points(case["n"], np.random.default_rng(seed))
        P = _bf16(_params(seed)).requires_grad_(True)
        loss = torch.mean((_forward(P, torch.from_numpy(x).double()) - torch.from_numpy(y).double()) ** 2)
        (grad,) = torch.autograd.grad(loss, P)
        return {"loss": np.array([float(loss.detach())]), "grad": grad.numpy()}
    if kind == "surface":
        sx, sy, _ = _surface(case, seed)
        w2 = 0.0
        for s in (sx, sy):
            h = np.concatenate([[0], np.cumsum(2 * s.astype(np.int64) - 1)[:-1]])
            w2 += float(np.var(h.astype(np.float64)))
        return {"w2": np.array([w2]), "S1": None, "S2": None, "heights": None, "slopes": None}
    return None
