#!/usr/bin/env python
"""Benchmark of the GB300 octahedron KPZ engine.

Workload (one step): the L = 2^16 job -- flat checkerboard start, p = 1, q = 0,
2000 Monte Carlo steps (sweeps of L^2 attempts each) with the exact width W^2
sampled at log-spaced times, through the C ABI of include/kpz.h. Metric:
site-update attempts per second (Kelling et al., arXiv:1204.5072, Sec. 4
report updates per second). One JSON line on stdout (rank 0).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference]

Besides `value` (lattice resident in HBM) the line carries `e2e` (the same job
with the start surface uploaded from pinned host memory and the final one read
back, per-part times and the bare pinned-copy bandwidth beside it), `roofline`
(the sweep kernel against the integer-logic pipe, with the HBM view, the
measured pipe peak and the DRAM traffic of the committed ncu capture),
`roofline_general` (the same kernel at p = 0.95, q = 0.05, the acceptance
path), `cpu_baseline` / `cpu_all_cores` / `cpu_rsu` (the oracle on a bounded
sample), `clocks`, `gpu_launches`, `batch` (the 512-realisation batched
workload at its 10^5-sweep cap in one persistent launch, with construction-free
baselines -- one launch per realisation, one lattice after another -- on a
stratified subset, per L bucket) and `surrogate` (trained on that batch's own
curves with one size held out; held-out errors, planned run lengths against
4 L^1.6, saturation times).

`--impl reference` times the CPU oracle (the plain single-threaded
restatement of the same schedule) on a bounded sample of the workload.
Under torchrun every rank runs its own independent realisation (sample =
rank): the path has no exchange step, so the scaling is weak and replica-only.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time
import warnings

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from synth import inputs as I  # noqa: E402

METRIC = "KPZ site-update attempts/s at L=2^16 (frac. of roofline); batched realisations/s"
UNIT = "attempts/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--L", type=int, default=I.L65536_2000.L)
    ap.add_argument("--mcs", type=int, default=I.L65536_2000.mcs)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--cpu-sample-mcs", type=int, default=100)
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--batch-cap", type=int, default=100_000)
    ap.add_argument("--batch-per-bucket", type=int, default=3)
    ap.add_argument("--batch-n", type=int, default=512)
    ap.add_argument("--batch-only", action="store_true",
                    help="profiling aid: run only the batched-ensemble section (no comparisons)")
    ap.add_argument("--no-surrogate", action="store_true")
    ap.add_argument("--no-general", action="store_true")
    ap.add_argument("--general-sweeps", type=int, default=100)
    return ap.parse_args()


def peaks():
    """(HBM GB/s, SM max MHz, source) from the measured peaks in MEASURED_PEAKS.json, else fallback figures."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), float(d.get("sm_max_mhz", 2070.0)), "measured"
    except Exception:
        return 6800.0, 2070.0, "fallback"


# ALU-pipe operations the algorithm needs per attempt at p = 1, q = 0, counted
# with three-input logic ops on 32 cells per word. Per round and cell-row word:
# 4 per quadrant site (the two neighbour-pair tests, their AND with the
# x-selection, the flip gated by the y-selection), 2 neighbour shifts and one
# dead-border mask: 19/32. Philox: 20 three-input xors per 128-bit block, 2 bits
# per attempt: 20/64. Window staging: one funnel shift per 32-site word and
# tile to align a loaded window (the store side is one wide multiply-add on
# the FMA pipe), 16 planes per 512 attempts: 1/32.
K_ALG_ALU = 19 / 32 + 20 / 64 + 1 / 32
ALU_LANES_PER_SM = 64   # integer logic pipe: 16 lanes per SM sub-partition per clock
# General rates (p, q strictly between 0 and 1): per round and word, the
# candidate test (all four neighbour bits equal: 2 per site), the selection and
# the minimum test (1 each per site), the per-row ORs of minima and candidates
# and the maxima (5), 2 neighbour shifts, the dead-border mask, the acceptance
# mask (2) and the flips (4): 30/32 instead of 19/32; plus the acceptance of
# the candidates (attempted site a local minimum or maximum, density C_CAND in
# the growth regime at p = 0.95: 0.176 minima + 0.202 maxima on oracle surfaces
# at L = 512, t = 100..2000), which a bit-serial comparison with the threshold
# decides with 2 random bits on average, each costing 20/128 Philox xors and
# 2/32 bit-sliced compare ops.
C_CAND = 0.378
K_ALG_ALU_GENERAL = 30 / 32 + 20 / 64 + 1 / 32 + C_CAND * 2 * (20 / 128 + 2 / 32)


# Files the sweep kernel is compiled from (their hash ties a profile to the source).
SWEEP_SOURCES = ("kpz_sweep.cu", "kpz_run.cuh", "kpz_rounds.cuh", "kpz_tilemem.cuh", "kpz_common.cuh",
                 "kpz_internal.h", "kpz_gridsync.cuh")


def sweep_source_sha():
    import hashlib
    src = b"".join(open(os.path.join(ROOT, "paper_1204_5072_gb300", "csrc", f), "rb").read()
                   for f in SWEEP_SOURCES)
    return hashlib.sha256(src).hexdigest()[:16]


def measured_traffic(L, profile="sweep_kernel_L65536.md"):
    """DRAM bytes per sweep launch from a committed ncu summary, if it was
    taken on this size and on the current kernel source; else None."""
    try:
        sha = sweep_source_sha()
        txt = open(os.path.join(ROOT, "profiles", profile)).read()
        fields = dict(ln.split(": ", 1) for ln in txt.splitlines() if ": " in ln and ln[:1].isalpha())
        if L == 65536 and fields.get("source_sha256") == sha:
            return float(fields["traffic_bytes_per_launch"])
    except Exception:
        pass
    return None


# --------------------------------------------------------------------------- #
class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.thread.join(timeout=2)

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 8:
                continue
            try:
                sm.append(float(f[0]))
                mx.append(float(f[1]))
            except ValueError:
                continue
            for n, v in zip(names, f[4:8]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# --------------------------------------------------------------------------- #
def cpu_baseline(L_full: int, mcs_sample: int):
    """The oracle, as it stands (single-threaded C), on a bounded sample of the
    workload: L = 1024 with the same schedule parameters, `mcs_sample` sweeps
    from the flat start and W^2 at the end."""
    from oracle import oracle as O
    L = 1024
    w = I.L65536_2000
    st = O.State.flat(L)
    t0 = time.perf_counter()
    st.run(mcs_sample, w.bx, w.by, w.p, w.q, w.seed, w.sample)
    st.w2()
    dt = time.perf_counter() - t0
    return {"value": mcs_sample * L * L / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"L={L} p={w.p} q={w.q} seed={w.seed}, {mcs_sample} MCS from the flat start "
                      f"+ W^2, 128x128 tiles (sub-run of the L={L_full} workload)",
            "seconds": dt}


def replica_sample(rank: int) -> int:
    """The realisation a rank runs under torchrun: sample = rank, i.e. its own
    Philox streams (the path has no exchange step; replicas only)."""
    return rank


def max_over_ranks(seconds: float, dist=None, device="cuda") -> float:
    """The slowest rank's time (the job ends when every rank has finished)."""
    if dist is None:
        return seconds
    import torch
    t = torch.tensor([seconds], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_value(world: int, steps: int, mcs: int, L: int, seconds: float) -> float:
    """Attempts/s of the whole job: every rank sweeps its own L x L lattice."""
    return float(world) * steps * mcs * L * L / seconds


def job_config(L, mcs, world):
    """The `config` of the benchmark job (both arms report the same one)."""
    w = I.L65536_2000
    n = len(I.sample_times(mcs))
    return {"workload": f"octahedron KPZ L={L} p=1 q=0 {mcs} MCS, W^2 at "
                        f"{n} log-spaced times, 1 realisation per GPU",
            "L": L, "p": w.p, "q": w.q, "mcs": mcs, "samples": n,
            "tile": "128x128, 4x4 cells", "seed": w.seed,
            "l2": "lattice (L^2/8 bytes = 512 MiB at L=2^16) larger than L2",
            "parallelism": f"replicas{world}"}


def cpu_all_cores(mcs_sample: int):
    """The oracle with the tiles of each sweep spread over every host core
    (bit-identical to the serial oracle), on the same L = 1024 sub-run."""
    from oracle import oracle as O
    L, w = 1024, I.L65536_2000
    cores = os.cpu_count() or 1
    st = O.State.flat(L)
    t0 = time.perf_counter()
    st.run_threads(mcs_sample, w.bx, w.by, w.p, w.q, w.seed, w.sample, threads=cores)
    st.w2()
    dt = time.perf_counter() - t0
    return {"value": mcs_sample * L * L / dt, "unit": UNIT, "cores": cores,
            "kind": "oracle, tiles of a sweep over all host threads",
            "sample": f"L={L}, {mcs_sample} MCS from the flat start + W^2", "seconds": dt}


def cpu_rsu(mcs_sample: int):
    """The oracle's random-sequential updates (one attempt at a uniformly random
    site at a time, no decomposition: the dynamics the decomposition
    approximates) on one core, L = 1024 from the flat start."""
    from oracle import oracle as O
    L, w = 1024, I.L65536_2000
    st = O.State.flat(L)
    t0 = time.perf_counter()
    st.rsu(mcs_sample, w.p, w.q, w.seed, w.sample)
    dt = time.perf_counter() - t0
    return {"value": mcs_sample * L * L / dt, "unit": UNIT, "cores": 1,
            "kind": "oracle, random-sequential updates",
            "sample": f"L={L}, {mcs_sample} MCS from the flat start", "seconds": dt}


# The paper's own update rates (order of magnitude from its text; its figures
# are not available): context for the GB300 numbers, not a target.
PAPER_CONTEXT = {"gpu_updates_per_s": 1e9,
                 "gpu_hardware": "Tesla C1060, Fermi C2050/C2070, Radeon HD5970/HD6970",
                 "cpu_updates_per_s": 1e7,
                 "cpu_hardware": "Opteron F8380, Core i5 430M, Core i7 920 (one core)",
                 "workload": "p = 1, q = 0, bit-coded lattice (Sec. 4)"}


def run_reference(a):
    """--impl reference: the CPU oracle timed on the host cores."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from oracle import oracle as O
    w = I.L65536_2000
    L, per_step = 1024, 4
    O.build()
    st = O.State.flat(L)
    for _ in range(a.warmup):
        st.run(per_step, w.bx, w.by, w.p, w.q, w.seed, w.sample)
    t0 = time.perf_counter()
    for _ in range(a.steps):
        st.run(per_step, w.bx, w.by, w.p, w.q, w.seed, w.sample)
        st.w2()
    dt = time.perf_counter() - t0
    value = a.steps * per_step * L * L / dt
    sample = (f"L={L} p={w.p} q={w.q} seed={w.seed}, {per_step} MCS + W^2 per step, "
              f"128x128 tiles (sub-run of the L={a.L} workload)")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": a.gpus, "steps": a.steps, "warmup": a.warmup,
            "ms_per_step": 1e3 * dt / a.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "u32", "data": "synthetic (flat checkerboard start)",
            "config": job_config(a.L, a.mcs, a.gpus),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------- #
def _timed(fn):
    """Wall time of fn() with the device idle on both sides."""
    import torch
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    fn()
    torch.cuda.synchronize()
    return time.perf_counter() - t0


def _per_lattice_run(eng, lat, n, times):
    """One realisation as a lattice of its own (kpz_run), W^2 at its sample times."""
    tp = 0
    for t in times:
        if t > n:
            break
        if t > tp:
            lat.run(t - tp)
        lat.roughness()
        tp = t


def batch_bench(eng, cap, seed=1, n_specs=512, per_bucket=3, compare=True):
    """Batched ensemble: the 512 realisations of the batched workload (L =
    2^{8..13} log-uniform, p ~ U[0.5, 1], q = 1 - p, run length min(4 L^1.6,
    cap)) in one persistent graph launch, created and autotuned before the
    clock. Against it, on a stratified subset (`per_bucket` realisations of
    each L, the first in seed order), every object also created before the
    clock: (i) one persistent launch per realisation and (ii) one Lattice per
    realisation (kpz_run between the samples), one after another, both with
    W^2 at the same times, each L bucket timed on its own beside the batched
    launch of the same bucket."""
    import numpy as np
    specs = [(s.L, s.p, s.q, seed, s.sample, min(s.mcs, cap)) for s in I.ensemble_specs(n_specs, seed=seed)]
    attempts = float(sum(L * L * n for L, _, _, _, _, n in specs))
    t0 = time.perf_counter()
    b = eng.Batch(specs, n_samples=64, autotune=True)
    create_s = time.perf_counter() - t0
    batched = _timed(b.run)
    times = [int(t) for t in b.times()]
    curves = b.w2()
    info = b.info()
    b.close()
    n = len(specs)
    out = {"metric": "batched realisations/s", "value": n / batched, "unit": "realisations/s",
           "attempts_per_s": attempts / batched, "seconds": batched, "attempts": attempts,
           "workload": f"{n} realisations, L=2^(8..13) log-uniform, p~U[0.5,1], q=1-p, "
                       f"T=min(ceil(4 L^1.6), {cap}) MCS, W^2 at the common log-spaced times (seed {seed})",
           "tuning": {k: info[k] for k in ("run", "warps_per_cta", "ctas_per_sm", "grid", "graph", "tile_y")},
           "create_and_autotune_s": create_s}
    result = {"specs": specs, "times": np.array(times), "w2": curves}
    if not compare:
        return out, result
    buckets = {}
    for sp in specs:
        if len(buckets.setdefault(sp[0], [])) < per_bucket:
            buckets[sp[0]].append(sp)
    sub = [sp for L in sorted(buckets) for sp in buckets[L]]
    rows = {}
    tot = {"batched": 0.0, "per_realisation": 0.0, "per_lattice": 0.0}
    bsub = eng.Batch(sub, n_samples=64, autotune=True)
    t_sub = _timed(bsub.run)
    bsub.close()
    for L in sorted(buckets):
        grp = buckets[L]
        one_b = eng.Batch(grp, n_samples=64, autotune=True)
        singles = [eng.Batch([sp], n_samples=64, autotune=True) for sp in grp]
        lats = [eng.Lattice(sp[0], sp[1], sp[2], seed=sp[3], sample=sp[4]) for sp in grp]
        tb = _timed(one_b.run)
        tr = _timed(lambda: [x.run() for x in singles])
        ts = _timed(lambda: [_per_lattice_run(eng, lat, sp[5], times) for lat, sp in zip(lats, grp)])
        for x in [one_b, *singles, *lats]:
            x.close()
        k = len(grp)
        rows[f"L{L}"] = {"n": k, "mcs": [sp[5] for sp in grp],
                         "batched_real_per_s": k / tb, "per_realisation_real_per_s": k / tr,
                         "per_lattice_real_per_s": k / ts,
                         "speedup_vs_per_realisation": tr / tb, "speedup_vs_per_lattice": ts / tb}
        tot["batched"] += tb
        tot["per_realisation"] += tr
        tot["per_lattice"] += ts
    k = len(sub)
    out["subset"] = {"workload": f"{per_bucket} realisations per L bucket ({k} in all), same specs, "
                                 f"every Batch/Lattice created (and autotuned) before its clock",
                     "batched_one_launch": {"value": k / t_sub, "seconds": t_sub},
                     "vs_launch_per_realisation": {"value": k / tot["per_realisation"],
                                                   "seconds": tot["per_realisation"],
                                                   "speedup": tot["per_realisation"] / t_sub},
                     "vs_lattice_per_realisation": {"value": k / tot["per_lattice"], "seconds": tot["per_lattice"],
                                             "speedup": tot["per_lattice"] / t_sub},
                     "per_bucket": rows}
    return out, result


def surrogate_bench(eng, full, cap, held_L=1024, factor=2.0):
    """Surrogate trained by the engine's kernels on the batched workload's own
    W^2 curves (`full`: the 512 realisations just simulated), with every
    realisation of size held_L left out; its error against fresh simulated
    ensembles at held-out (L, p) -- including L = held_L, absent from
    training -- and the run lengths it plans (min(cap, factor t_x)) against
    the fixed rule min(cap, 4 L^1.6)."""
    import math
    import numpy as np
    from paper_1204_5072_gb300 import surrogate as S

    def heur(L):
        return int(min(math.ceil(4 * L ** 1.6), cap))

    specs, times, w2 = full["specs"], full["times"], full["w2"]
    keep = [i for i, sp in enumerate(specs) if sp[0] != held_L]
    t0 = time.perf_counter()
    sur = S.Surrogate.fit([specs[i] for i in keep], times, w2[keep], epochs=300, batch=128, lr=3e-3, seed=1,
                          p_bin=0.05)
    train_s = time.perf_counter() - t0
    n_train = int(sum(((times > 0) & (times <= specs[i][5])).sum() for i in keep))

    def ens(L, p, n_real, T):
        b = eng.Batch([(L, p, 1 - p, 77, 9000 + k, T) for k in range(n_real)], n_samples=48)
        b.run()
        t, w = b.times(), b.w2()
        b.close()
        with warnings.catch_warnings():
            warnings.simplefilter("ignore", RuntimeWarning)
            return t, np.nanmean(w, axis=0)

    held = {}
    t0 = time.perf_counter()
    for L, n_real, T in [(256, 64, heur(256)), (held_L, 24, heur(held_L)), (4096, 6, min(heur(4096), 20_000))]:
        for p in (0.6, 0.9):
            t, m = ens(L, p, n_real, T)
            sel = (t >= 1) & (t <= T) & np.isfinite(m)
            err = float(np.mean(np.abs(sur.w2(L, t[sel], p, 1 - p) / m[sel] - 1)))
            held[f"L{L}_p{p}"] = {"mean_rel_error": err, "realisations": n_real, "mcs": T,
                                  "in_training": L != held_L}
    sim_s = time.perf_counter() - t0
    # Run lengths for the batched workload's own specs.
    planned = sur.plan(specs, factor=factor, cap=cap)
    fixed_att = sum(L * L * heur(L) for (L, *_r) in specs)
    plan_att = sum(sp[0] * sp[0] * sp[5] for sp in planned)
    Ls = [256, 512, 1024, 2048, 4096, 8192]
    # t_x is searched only inside the trained time range (t <= cap): for the
    # sizes that do not saturate under the cap the network's value is a lower
    # bound, and the power law through L = 256 and 512 extrapolates instead.
    tx, _ = sur.t_x_fit(Ls, 0.75, 0.25, t_max=cap)
    tx_small, z = sur.t_x_fit([256, 512], 0.75, 0.25, t_max=cap)
    # Plateau reached by the planned runs (sizes that saturate under the cap).
    plateau = {}
    for L in (256, 512):
        for p in (0.6, 0.9):
            Tp = int(min(cap, math.ceil(factor * sur.t_sat(L, p, 1 - p, t_max=cap))))
            runs = {}
            for tag, T, ns in (("fixed", heur(L), 96), ("planned", Tp, 48)):
                bb = eng.Batch([(L, p, 1 - p, 78, 9500 + k, T) for k in range(128)], n_samples=ns)
                bb.run()
                runs[tag] = (bb.times(), bb.w2())
                bb.close()
            tl, wl = runs["fixed"]
            tp_, wp = runs["planned"]
            per_real = wl[:, (tl >= 0.5 * heur(L)) & (tl <= heur(L))].mean(axis=1)
            end_w = wp[:, int(np.searchsorted(tp_, Tp))]
            ref = float(per_real.mean())
            plateau[f"L{L}_p{p}"] = {"planned_mcs": Tp, "fixed_mcs": heur(L),
                                     "end_over_plateau": float(end_w.mean()) / ref,
                                     "std_error": float(np.sqrt(end_w.var(ddof=1) / 128 +
                                                                per_real.var(ddof=1) / 128)) / ref}
    sur.close()
    return {"trained_on": f"{len(keep)} curves of the batched workload ({n_train} (L, t, p) points), "
                          f"averaged into ensemble means over p bins of 0.05, L={held_L} left out",
            "held_out": held, "max_mean_rel_error": max(v["mean_rel_error"] for v in held.values()),
            "planned_attempts_frac_of_fixed_rule": plan_att / fixed_att,
            "planned_vs_fixed_by_L": {f"L{L}": [int(np.mean([sp[5] for sp in planned if sp[0] == L])), heur(L)]
                                      for L in Ls},
            "plateau_check": plateau,
            "t_x_pred": {f"L{L}": float(v) for L, v in zip(Ls, tx)},
            "t_x_powerlaw_from_L256_512": {"z": z, "extrapolated": {f"L{L}": float(tx_small[1] * (L / 512) ** z)
                                                                   for L in Ls[2:]}},
            "train_s": train_s, "simulate_s": sim_s}


# --------------------------------------------------------------------------- #
def main():
    a = parse()
    if a.impl == "reference":
        run_reference(a)
        return

    import numpy as np
    import torch

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    import __graft_entry__
    __graft_entry__.build()
    import paper_1204_5072_gb300 as eng
    from paper_1204_5072_gb300._lib import launch_count
    if a.batch_only:   # profiling aid: the batched-ensemble section alone
        if rank == 0:
            print(json.dumps(batch_bench(eng, a.batch_cap, n_specs=a.batch_n, compare=False)[0]), flush=True)
        return

    w = I.L65536_2000
    L, mcs = a.L, a.mcs
    times = I.sample_times(mcs)
    stream = torch.cuda.current_stream()
    lat = eng.Lattice(L, w.p, w.q, seed=w.seed, sample=replica_sample(rank))

    sweep_events = []  # (start, end, n_sweeps) on the engine's stream

    def job(record=False):
        lat.reset()
        t_prev = 0
        rough = []
        for t in times:
            n = t - t_prev
            if n:
                if record:
                    e0 = torch.cuda.Event(enable_timing=True)
                    e1 = torch.cuda.Event(enable_timing=True)
                    e0.record(stream)
                lat.run(n)
                if record:
                    e1.record(stream)
                    sweep_events.append((e0, e1, n))
            rough.append(lat.roughness())
            t_prev = t
        return rough

    def barrier():
        if dist:
            dist.barrier()
        torch.cuda.synchronize()

    for _ in range(max(a.warmup, 3)):
        job()
    barrier()
    launches0 = launch_count()
    with ClockSampler(local) as clk:
        t_start = torch.cuda.Event(enable_timing=True)
        t_end = torch.cuda.Event(enable_timing=True)
        t_start.record(stream)
        for _ in range(a.steps):
            rough = job(record=True)
        t_end.record(stream)
        torch.cuda.synchronize()
    launches = launch_count() - launches0
    elapsed = max_over_ranks(t_start.elapsed_time(t_end) / 1e3, dist)
    attempts = float(world) * a.steps * mcs * L * L
    value = whole_job_value(world, a.steps, mcs, L, elapsed)
    sweep_ms = sum(e0.elapsed_time(e1) for e0, e1, _ in sweep_events)
    n_sweeps = sum(n for _, _, n in sweep_events)
    per_sweep_s = sweep_ms / 1e3 / n_sweeps

    # Roofline of the sweep kernel. The state is one bit per site, read and
    # written once per sweep (0.25 B/attempt); the integer-logic pipe binds
    # first: K_ALG_ALU ops per attempt against 152 SMs x 64 lanes x clock.
    hbm_peak, sm_mhz, peak_kind = peaks()
    sms = torch.cuda.get_device_properties(local).multi_processor_count
    alg_bytes = 0.25 * L * L
    alu_peak = sms * ALU_LANES_PER_SM * sm_mhz * 1e6 / 1e12          # Top/s
    alu_achieved = K_ALG_ALU * L * L / per_sweep_s / 1e12
    hbm_achieved = alg_bytes / per_sweep_s / 1e9
    roofline = {"bound": "alu", "achieved": alu_achieved, "peak": alu_peak, "unit": "Top/s",
                "frac": alu_achieved / alu_peak, "traffic": measured_traffic(L),
                "kernel": "sweep_kernel", "alg_ops_per_attempt": K_ALG_ALU,
                "launch_ms": per_sweep_s * 1e3,
                "peak_source": f"{sms} SMs x {ALU_LANES_PER_SM} ALU lanes x {sm_mhz:.0f} MHz ({peak_kind} clock)",
                "hbm": {"achieved": hbm_achieved, "peak": hbm_peak, "unit": "GB/s",
                        "frac": hbm_achieved / hbm_peak, "alg_bytes_per_launch": alg_bytes,
                        "peak_source": f"{peak_kind} hbm_gbs"}}
    # The derived ALU peak checked by the engine's own LOP3 throughput probe
    # (outside the timed region).
    try:
        probe = eng._lib.alu_peak()
        roofline["peak_probe"] = {"value": probe["lane_ops_per_s"] / 1e12, "unit": "Top/s",
                                  "of_derived": probe["lane_ops_per_s"] / 1e12 / alu_peak,
                                  "source": "kpz_alu_peak: one wave of independent LOP3 chains"}
    except Exception as exc:   # report, do not hide
        roofline["peak_probe"] = {"error": str(exc)}

    # The same kernel at general rates (p = 0.95, q = 0.05: acceptance draws),
    # the path of the batched workload; CUDA events on the engine's stream.
    roofline_general = None
    if not a.no_general:
        lat_g = eng.Lattice(L, 0.95, 0.05, seed=w.seed, sample=replica_sample(rank))
        lat_g.run(5)
        torch.cuda.synchronize()
        ng = max(10, min(200, a.general_sweeps))
        g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        g0.record(stream)
        lat_g.run(ng)
        g1.record(stream)
        torch.cuda.synchronize()
        per_g = g0.elapsed_time(g1) / 1e3 / ng
        lat_g.close()
        ach = K_ALG_ALU_GENERAL * L * L / per_g / 1e12
        roofline_general = {"bound": "alu", "achieved": ach, "peak": alu_peak, "unit": "Top/s",
                            "frac": ach / alu_peak,
                            "traffic": measured_traffic(L, "sweep_kernel_general_L65536.md"),
                            "kernel": "sweep_chain_kernel (general rates)", "p": 0.95, "q": 0.05,
                            "alg_ops_per_attempt": K_ALG_ALU_GENERAL, "candidate_density": C_CAND,
                            "launch_ms": per_g * 1e3, "sweeps_timed": ng, "start": "t = 5 from the flat start",
                            "attempts_per_s": L * L / per_g,
                            "hbm": {"achieved": alg_bytes / per_g / 1e9, "peak": hbm_peak, "unit": "GB/s",
                                    "frac": alg_bytes / per_g / 1e9 / hbm_peak}}

    # End to end through the C ABI with host buffers: upload the start state
    # from pinned memory, run the job with W^2 sampling, read the final lattice.
    e2e = None
    if not a.no_e2e:
        nwords = L * L // 16
        h_in = torch.empty(nwords, dtype=torch.int32, pin_memory=True)
        h_out = torch.empty(nwords, dtype=torch.int32, pin_memory=True)
        host_in = h_in.numpy().view(np.uint32)
        host_in.reshape(L, L // 16)[0::2] = 0x33333333
        host_in.reshape(L, L // 16)[1::2] = 0xCCCCCCCC
        host_out = h_out.numpy().view(np.uint32)

        parts = []   # host clock at the boundaries; every call returns after its stream work

        def e2e_step():
            c0 = time.perf_counter()
            lat.set_slopes(host_in, h00=0, t=0)
            c1 = time.perf_counter()
            t_prev = 0
            for t in times:
                if t - t_prev:
                    lat.run(t - t_prev)
                lat.roughness()
                t_prev = t
            c2 = time.perf_counter()
            lat.slopes_into(host_out)
            parts.append((c1 - c0, c2 - c1, time.perf_counter() - c2))

        e2e_step()
        barrier()
        parts.clear()
        t0 = time.perf_counter()
        for _ in range(a.steps):
            e2e_step()
        barrier()
        e2e_dt = max_over_ranks(time.perf_counter() - t0, dist)
        final_serial = host_out.copy()   # the bare-copy probe below overwrites h_out
        med = np.median(np.array(parts), axis=0) * 1e3
        # The bare pinned-memory copies of the same buffers in this process, for
        # reading the import/export parts (host links differ from box to box).
        dev_tmp = torch.empty(nwords, dtype=torch.int32, device="cuda")
        link = []
        for _ in range(2):
            torch.cuda.synchronize()
            c0 = time.perf_counter()
            dev_tmp.copy_(h_in, non_blocking=True)
            torch.cuda.synchronize()
            c1 = time.perf_counter()
            h_out.copy_(dev_tmp, non_blocking=True)
            torch.cuda.synchronize()
            link.append((c1 - c0, time.perf_counter() - c1))
        del dev_tmp
        best = np.min(np.array(link), axis=0)
        serial = {"value": attempts / e2e_dt, "unit": UNIT, "seconds": e2e_dt,
                  "parts_ms": {"import": round(float(med[0]), 2), "job": round(float(med[1]), 2),
                               "export": round(float(med[2]), 2)}}

        # Pipelined: two lattices on their own streams, each step of a lattice
        # (import, job, export) issued by its own host thread, so one lattice's
        # transfers overlap the other's sweeps; every step still copies its
        # start surface in and its final surface out inside the timed region.
        import threading as _th
        pipes = []
        for _ in range(2):
            st_ = torch.cuda.Stream()
            hi = torch.empty(nwords, dtype=torch.int32, pin_memory=True)
            hi.copy_(h_in)
            ho = torch.empty(nwords, dtype=torch.int32, pin_memory=True)
            lx = eng.Lattice(L, w.p, w.q, seed=w.seed, sample=replica_sample(rank), stream=st_.cuda_stream)
            pipes.append((st_, lx, hi.numpy().view(np.uint32), ho.numpy().view(np.uint32), hi, ho))

        def pipe_step(lx, hin, hout):
            lx.set_slopes(hin, h00=0, t=0)
            tp = 0
            for t in times:
                if t - tp:
                    lx.run(t - tp)
                lx.roughness()
                tp = t
            lx.slopes_into(hout)

        def pipe_worker(k, nsteps):
            _, lx, hin, hout, _, _ = pipes[k]
            for _ in range(nsteps):
                pipe_step(lx, hin, hout)

        for k in range(2):                      # warm-up of both pipes
            pipe_step(*pipes[k][1:4])
        barrier()
        t0 = time.perf_counter()
        ths = [_th.Thread(target=pipe_worker, args=(k, (a.steps + 1 - k) // 2)) for k in range(2)]
        for th in ths:
            th.start()
        for th in ths:
            th.join()
        barrier()
        pipe_dt = max_over_ranks(time.perf_counter() - t0, dist)
        ok = all(np.array_equal(pipes[k][3], final_serial) for k in range(2))
        for pp in pipes:
            pp[1].close()
        del pipes
        e2e = {"value": attempts / pipe_dt, "unit": UNIT, "h2d_bytes_per_step": nwords * 4,
               "d2h_bytes_per_step": nwords * 4 + len(times) * 48,
               "mode": "two lattices on their own streams, steps alternating between two host threads: "
                       "one lattice's import and export overlap the other's sweeps",
               "seconds": pipe_dt, "same_result_as_serial": bool(ok),
               "serial": serial,
               "bare_copy_gbs": {"h2d": round(nwords * 4 / best[0] / 1e9, 1),
                                 "d2h": round(nwords * 4 / best[1] / 1e9, 1)}}

    cpu = cpu_mt = cpu_seq = None
    if rank == 0 and world == 1 and not a.no_cpu:
        cpu = cpu_baseline(L, a.cpu_sample_mcs)
        cpu_mt = cpu_all_cores(max(10, a.cpu_sample_mcs // 2))
        cpu_seq = cpu_rsu(max(4, a.cpu_sample_mcs // 10))
    batch = sur = None
    if not (a.no_batch or world > 1):
        batch, full = batch_bench(eng, a.batch_cap, n_specs=a.batch_n, per_bucket=a.batch_per_bucket)
        if not a.no_surrogate:
            sur = surrogate_bench(eng, full, a.batch_cap)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": a.steps,
                "warmup": max(a.warmup, 3), "ms_per_step": 1e3 * elapsed / a.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
                "data": "synthetic (flat checkerboard start, p=1 q=0)",
                "config": job_config(L, mcs, world),
                "roofline": roofline, "roofline_general": roofline_general, "cpu_baseline": cpu, "cpu_all_cores": cpu_mt, "cpu_rsu": cpu_seq,
                "paper_context": PAPER_CONTEXT, "e2e": e2e,
                "clocks": clk.summary(), "gpu_launches": launches,
                "w2_final": rough[-1]["w2"], "batch": batch, "surrogate": sur}
        print(json.dumps(line), flush=True)
    lat.close()
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
