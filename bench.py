"""Benchmark of the coupled LB phase-field step on GB300.

Default workload: 2D 1024 x 1024, flow D2Q9 BGK tau_f = 0.6 coupled to the
phase-field and solute D2Q9 lattices, inflow u = 0.01 on the left,
zero-gradient outflow, periodic y, seed of radius 16 at x = 300, U0 = 0.4,
5-fold anisotropy of strength 0.03, FP32.  One benchmark step is one LB time
step over the whole grid; the metric is MLUPS (million node updates per
second) with the HBM roofline of the step kernel beside it.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--workload c1|c2|c2_fp16|c3|c3s|c3_fp16|c3s_fp16|c3_bf16|c4|c4s|c5|c5net|f1|f2|f3|
                              f3_3d|f3_3ds]

Workloads f1 (the crystal-shape measurement with a hexagonal seed), f2 (a
baffle of solid nodes in front of the inlet) and f3 (the central Hermite MRT
flow collision) run the C2 problem with those parts; f3_3d runs the C3 problem
with the central Hermite MRT (f3_3ds: its 128^3 case for profiler captures).

Workload c5 times the learned block propagator (a U-Net trained on the GPU
on trajectories of this solver, judged by and falling back to the LB)
against the plain LB on a held-out problem; --steps is then the number of
LB-equivalent steps timed.

Multi-GPU: a single grid is not sharded (one grid per GPU), so N GPUs run N
independent replicas ("replicas only", weak scaling).  The batched sweeps (c4,
c4s) are sharded: rank r of N advances every N-th instance of a sweep of
N x batch instances, with no exchange between ranks (weak scaling); the
whole-job rate counts the nodes of all shards.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)


def sources(*units):
    """The units and every file of the library that they include, in a fixed order."""
    found = []
    todo = list(units)
    while todo:
        f = todo.pop(0)
        if f in found:
            continue
        found.append(f)
        text = open(os.path.join(ROOT, "paper_2206_02145_gb300", "csrc", f)).read()
        todo += [i for i in re.findall(r'^#include "([^"]+)"', text, re.M) if "/" not in i]
    return found


# the files each timed kernel is compiled from (a committed profile's counters
# stand only while their digest is unchanged)
SRC_2D = sources("step2d.cu")
SRC_3D = sources("step3d.cu")
SRC_BATCH = sources("batch2d.cu", "batch2d_fp32.cu", "batch2d_fp16.cu", "batch2d_bf16.cu")
SRC_CONV = sources("conv_tc.cu")
SRC_FACETS = sources("facets.cu")

# bytes each node moves through HBM per step (populations read + written,
# phi(t-1) read, phi(t) written)
WORKLOADS = {
    "c2": dict(desc="2D 1024x1024 coupled LB (D2Q9 flow + solute + phase field), inflow 0.01, "
                    "seed R=16 at x=300, U0=0.4, 5-fold eps 0.03",
               dim=2, nx=1024, ny=1024, nz=1, flow=1, fold=5, eps=0.03, bc=(1, 0, 0),
               u_in=0.01, U_in=0.4, seed=(300.0, 512.0, 0.0, 16.0, 0.4, 0.01, 1),
               storage="fp32", kernel="step2d_tma_kernel", src=SRC_2D, fp16_compare=True,
               sample=dict(nx=256, ny=256, seed=(75.0, 128.0, 0.0, 16.0, 0.4, 0.01, 1))),
    "c2_fp16": dict(base="c2", storage="fp16", fp16_compare=False),
    "f2": dict(base="c2", desc_note=True,
               desc="2D 1024x1024 coupled LB, inflow 0.01, seed R=16 at x=300, U0=0.4, 5-fold "
                    "eps 0.03, with a baffle of solid nodes 4 lu thick and 320 lu long at x=150 "
                    "in front of the inlet (dimensions invented: the paper shows its baffles "
                    "only in a figure)",
               baffle=dict(x0=150, y0=352, y1=672, w=4), kernel="step2d_tma_kernel_mask",
               sample=dict(nx=256, ny=256, seed=(75.0, 128.0, 0.0, 16.0, 0.4, 0.01, 1),
                           baffle=dict(x0=37, y0=88, y1=168, w=1))),
    "f3": dict(base="c2", desc_note=True,
               desc="2D 1024x1024 coupled LB, inflow 0.01, seed R=16 at x=300, U0=0.4, 5-fold "
                    "eps 0.03, the flow colliding by the central Hermite MRT (trace of the "
                    "second-order and the third/fourth-order central moments relaxed at 1)",
               collision=1, kernel="step2d_tma_kernel_chm"),
    "f1": dict(desc="2D 1024x1024 coupled LB, inflow 0.01, hexagonal seed (perimeter 120 lu, "
                    "side normals at 0.1 + pi/6 + k pi/3) at x=300, U0=0.4, 6-fold eps 0.03 at "
                    "theta0 0.1; crystal shape (side lengths, centre, Q, aspect ratio) measured "
                    "every 1000 steps, growth rates and R^2 fitted",
               dim=2, nx=1024, ny=1024, nz=1, flow=1, fold=6, eps=0.03, theta0=0.1,
               bc=(1, 0, 0), u_in=0.01, U_in=0.4, every=1000,
               polygon=dict(cx=300.0, cy=512.0, perimeter=120.0, u0=0.4, noise=0.01, seed=1),
               storage="fp32", kernel="step2d_tma_kernel", src=SRC_2D,
               sample=dict(nx=256, ny=256,
                           polygon=dict(cx=75.0, cy=128.0, perimeter=120.0, u0=0.4,
                                        noise=0.01, seed=1))),
    "c1": dict(desc="2D 128x128 periodic, no flow (phase field + solute D2Q9), U0=0.3, R=8, "
                    "4-fold eps 0.05",
               dim=2, nx=128, ny=128, nz=1, flow=0, fold=4, eps=0.05, bc=(0, 0, 0), u_in=0.0,
               U_in=0.0, seed=(64.0, 64.0, 0.0, 8.0, 0.3, 0.01, 1), storage="fp32",
               kernel="step2d_tma_kernel", src=SRC_2D,
               sample=dict(nx=128, ny=128, seed=(64.0, 64.0, 0.0, 8.0, 0.3, 0.01, 1))),
    "c3": dict(desc="3D 256^3 coupled LB (D3Q19 flow, D3Q7 solute and phase field), cubic eps "
                    "0.04, sphere R=12, U0=0.3, inflow 0.005",
               dim=3, nx=256, ny=256, nz=256, flow=1, fold=0, eps=0.04, bc=(1, 0, 0),
               u_in=0.005, U_in=0.3, seed=(128.0, 128.0, 128.0, 12.0, 0.3, 0.01, 1),
               storage="fp32", kernel="step3d_column_kernel", src=SRC_3D,
               sample=dict(nx=48, ny=48, nz=48, seed=(24.0, 24.0, 24.0, 12.0, 0.3, 0.01, 1))),
    "c3_fp16": dict(base="c3", storage="fp16"),
    "c3s": dict(base="c3", nx=128, ny=128, nz=128, seed=(64.0, 64.0, 64.0, 12.0, 0.3, 0.01, 1),
                desc="3D 128^3 case of c3 for profiler captures (D3Q19 flow, D3Q7 solute and "
                     "phase field), cubic eps 0.04, sphere R=12, U0=0.3, inflow 0.005",
                desc_note="FP32"),
    "c3s_fp16": dict(base="c3", nx=128, ny=128, nz=128, storage="fp16",
                     seed=(64.0, 64.0, 64.0, 12.0, 0.3, 0.01, 1),
                     desc="3D 128^3 case of c3_fp16 for profiler captures (D3Q19 flow, D3Q7 "
                          "solute and phase field), cubic eps 0.04, sphere R=12, U0=0.3, inflow "
                          "0.005, FP16 shifted storage", desc_note=True),
    "c3_bf16": dict(base="c3", storage="bf16"),
    "f3_3d": dict(base="c3", desc_note=True,
                  desc="3D 256^3 coupled LB (D3Q19 flow, D3Q7 solute and phase field), cubic "
                       "eps 0.04, sphere R=12, U0=0.3, inflow 0.005, the flow colliding by the "
                       "central Hermite MRT (trace of the second-order and the third/fourth-"
                       "order central moments relaxed at 1)",
                  collision=1, kernel="step3d_column_kernel_chm"),
    "f3_3ds": dict(base="c3", nx=128, ny=128, nz=128, collision=1,
                   kernel="step3d_column_kernel_chm",
                   seed=(64.0, 64.0, 64.0, 12.0, 0.3, 0.01, 1), desc_note=True,
                   desc="3D 128^3 case of f3_3d for profiler captures (D3Q19 flow colliding by "
                        "the central Hermite MRT, D3Q7 solute and phase field), cubic eps 0.04, "
                        "sphere R=12, U0=0.3, inflow 0.005"),
    "c4": dict(desc="batched sweep: 64 2D coupled instances in one persistent launch per step "
                    "(sides U{256..768}, U0~U[0.1,0.6], R~U[4,24], u_in~U[0,0.02], fold 4 or 5, "
                    "eps~U[0.02,0.06]; seed 4), FP16 shifted storage",
               dim=2, nx=512, ny=512, nz=1, flow=1, fold=5, eps=0.04, bc=(1, 0, 0), u_in=0.01,
               U_in=0.35, storage="fp16", kernel="step2d_batch_kernel", src=SRC_BATCH,
               batch=64, sweep_seed=4,
               sample=dict(nx=256, ny=256, seed=(77.0, 128.0, 0.0, 12.0, 0.35, 0.01, 1))),
    "c4s": dict(base="c4", batch=256, sides=(32, 128),
                desc="batched sweep of small instances: 256 2D coupled instances in one "
                     "persistent launch per step (sides U{32..128}, U0~U[0.1,0.6], "
                     "R~U[4,min(24,n/5)], u_in~U[0,0.02], fold 4 or 5, eps~U[0.02,0.06]; "
                     "seed 4), FP16 shifted storage", desc_note="small instances",
                kernel="step2d_batch_kernel_small"),
    "c5": dict(desc="learned block propagator on 2D 512x512 closed channels (periodic x, walls y, "
                    "body-force Poiseuille flow u_max~U[0,0.01], U0~U[0.25,0.45], R~U[6,16], "
                    "fold 4 or 5, eps~U[0.02,0.05]): BF16 U-Net 32/64/128/256 channels trained "
                    "on the GPU on 2000 LB pairs from 50 sampled problems (mirror "
                    "augmentation; Adam 8000 steps at 2.5e-4 for 50-step blocks, 4000 at 5e-4 "
                    "for 200), blocks of 50 LB steps (and 200 beside them), LB judge every "
                    "8th block, fallback at drift > 1e-3 or interface error > 1 lu; held-out "
                    "problem; FP32 LB",
               dim=2, nx=512, ny=512, nz=1, flow=1, fold=5, eps=0.03, bc=(0, 2, 0), u_in=0.0,
               U_in=0.0, storage="fp32", kernel="conv3x3_tc_kernel", src=SRC_CONV,
               # training recipe per block length (Adam steps, learning rate): the
               # 50-step network needs the smaller rate (at 5e-4 its small
               # per-block bias accumulates to lattice units over 400 blocks)
               surrogate=dict(blocks=(50, 200), judge_every=8, traj=50, t_end=20000,
                              every=500, crop=256, batch=8, start=1000, min_steps=20000,
                              val_steps=5000, val_tol=0.5, val_seeds=3, iface_rel_tol=0.9,
                              recipe={50: (8000, 2.5e-4), 200: (4000, 5e-4)}),
               sample=dict(nx=256, ny=256, channel=True)),
    "c5net": dict(desc="the c5 network alone: BF16 U-Net 32/64/128/256 channels on a 512x512 "
                       "sample (4 -> 4 channels, random weights): forward passes, then "
                       "training steps (forward, backward, Adam)",
                  dim=2, nx=512, ny=512, nz=1, flow=1, fold=5, eps=0.03, bc=(0, 2, 0),
                  u_in=0.0, U_in=0.0, storage="fp32", kernel="conv3x3_tc_kernel",
                  src=SRC_CONV, network=dict(batch=1),
                  sample=dict(nx=256, ny=256, channel=True)),
}


def sweep_members(count: int, seed: int, lo: int = 256, hi: int = 768):
    """Seeded uneven parametric sweep (the synthetic stand-in for the paper's
    supersaturation x seed-size x inflow studies): square sides U{lo..hi},
    U0 ~ U[0.1, 0.6], seed radius ~ U[4, min(24, n/5)], inflow ~ U[0, 0.02],
    fold 4 or 5, anisotropy ~ U[0.02, 0.06]; seed at (0.3 n, 0.5 n)."""
    import numpy as np
    rng = np.random.default_rng(seed)
    params, seeds = [], []
    for i in range(count):
        n = int(rng.integers(lo, hi + 1))
        u0 = float(rng.uniform(0.1, 0.6))
        r = float(rng.uniform(4, min(24, n / 5)))
        params.append(dict(dim=2, nx=n, ny=n, flow=1, fold=int(rng.choice([4, 5])),
                           eps_aniso=float(rng.uniform(0.02, 0.06)), bc=(1, 0, 0),
                           u_inlet=float(rng.uniform(0.0, 0.02)), u0_inlet=u0))
        seeds.append((0.3 * n, 0.5 * n, 0.0, r, u0, 0.01, 1000 + i))
    return params, seeds
ELEM = {"fp32": 4, "fp64": 8, "fp16": 2, "bf16": 2}


def shard(members, rank: int, world: int):
    """The members of a sweep that rank `rank` of `world` advances: every
    world-th one from its rank on (instances are independent: no exchange)."""
    params, seeds = members
    return params[rank::world], seeds[rank::world]


def lup_bytes(w, storage):
    """Algorithmic bytes of one node update of workload w with the given
    population storage: every population read and written once, the phi ring
    read and written, the solid mask read, and with 16-bit storage the per-node
    g reference (the node's own read, its neighbours' encoding reference read,
    the new one written)."""
    q = (9 if w["dim"] == 2 else 19) * w["flow"] + 2 * (9 if w["dim"] == 2 else 7)
    ring = 8 if storage == "fp64" else 4
    b = 2 * q * ELEM[storage] + 2 * ring
    if w.get("baffle"):
        b += 1  # the solid mask
    if ELEM[storage] == 2:
        b += 3 * 2
    return b


def workload(name, rank: int = 0, world: int = 1):
    """The workload's settings for rank `rank` of `world`.  nodes: the nodes
    this rank steps; nodes_all: those of all ranks (replicas of one grid, or
    the shards of a sweep of world x batch instances)."""
    w = dict(WORKLOADS[name])
    if "base" in w:
        b = dict(WORKLOADS[w.pop("base")])
        note = w.pop("desc_note", None)
        b.update(w)
        if not note:
            b["desc"] = b["desc"] + f", {b['storage'].upper()} shifted storage"
        w = b
    w["bytes_per_lup"] = lup_bytes(w, w["storage"])
    w["nodes"] = w["nx"] * w["ny"] * w["nz"]
    w["nodes_all"] = w["nodes"] * world
    if w.get("batch"):
        full = sweep_members(w["batch"] * world, w["sweep_seed"], *w.get("sides", (256, 768)))
        w["members"] = shard(full, rank, world)
        w["nodes"] = sum(p["nx"] * p["ny"] for p in w["members"][0])
        w["nodes_all"] = sum(p["nx"] * p["ny"] for p in full[0])
    return w


def lib_params(w, L, storage=None):
    return dict(dim=w["dim"], nx=w["nx"], ny=w["ny"], nz=w["nz"], bc=w["bc"], flow=w["flow"],
                storage={"fp32": L.FP32, "fp64": L.FP64, "fp16": L.FP16_SHIFTED,
                         "bf16": L.BF16_SHIFTED}[storage or w["storage"]],
                fold=w["fold"], eps_aniso=w["eps"], u_inlet=w["u_in"], u0_inlet=w["U_in"],
                theta0=w.get("theta0", 0.0), collision=w.get("collision", 0))


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        try:
            d = json.load(open(path))
            flat = {}

            def walk(o, pre=""):
                if isinstance(o, dict):
                    for k, v in o.items():
                        walk(v, pre + k + ".")
                else:
                    flat[pre[:-1]] = o
            walk(d)
            for k, v in flat.items():
                if re.search(r"hbm.*(gbs|gb_s|gbps)", k, re.I) and isinstance(v, (int, float)):
                    return float(v), "measured"
        except Exception:
            pass
    return 6800.0, "fallback"


def max_over_ranks(values, dist=None, device="cuda"):
    """The element-wise maximum of per-rank timings over all ranks (the job
    is as slow as its slowest replica); the values themselves without a
    process group.  device: where the reduction runs (cuda for NCCL, cpu for
    gloo)."""
    if dist is None:
        return [float(v) for v in values]
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t.tolist()]


def whole_job_rate(units_per_rank, world, seconds):
    """Whole-job throughput: the units all ranks processed over the slowest
    rank's time (weak scaling: every replica processes the same units)."""
    return units_per_rank * world / seconds


def iface_compare(d0, fast, plain, dim, min_growth=0.5):
    """The fast form's interface against the plain FP32 run from the same
    start: largest position difference over the axis rays (lattice units) and
    the relative growth-rate error per ray (rays that grew by > min_growth)."""
    n = 4 if dim == 2 else 6
    err, rel = [], []
    for r in range(n):
        a, b, c = fast[r], plain[r], d0[r]
        if a < 0 or b < 0 or c < 0:
            continue
        err.append(abs(a - b))
        g = b - c
        if abs(g) > min_growth:
            rel.append((a - c - g) / g)
    return (max(err) if err else None), rel


def source_digest(files):
    """sha256 over the concatenated sources a kernel is compiled from."""
    h = hashlib.sha256()
    for f in files:
        h.update(open(os.path.join(ROOT, "paper_2206_02145_gb300", "csrc", f), "rb").read())
    return h.hexdigest()


def measured_bf16():
    """Dense bf16 peak for a kernel timed on its own: the measured burst figure
    of MEASURED_PEAKS.json, else the 1.9 PFLOP/s fallback."""
    try:
        d = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
        v = d.get("bf16_tflops")
        if isinstance(v, (int, float)) and v > 0:
            return float(v), "measured"
    except Exception:
        pass
    return 1900.0, "fallback"


def profiled_traffic(w):
    """Per-launch DRAM bytes from the committed ncu summary of this kernel, or
    None when the kernel's sources changed since the counters were taken."""
    prof = os.path.join(ROOT, "profiles", f"{w['kernel']}_{w['nx']}_{w['storage']}.md")
    if not os.path.exists(prof):
        return None
    text = open(prof).read()
    mh = re.search(r"source_sha256[^:\n]*:\s*([0-9a-f]+)", text)
    mt = re.search(r"dram_bytes_per_launch:\s*([0-9.eE+]+)", text)
    if not (mh and mt):
        return None
    if source_digest(w["src"]) != mh.group(1):
        return None
    return float(mt.group(1))


class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled every 50 ms from before
    the warm-up to the end of the timed region; summary() keeps the samples
    taken inside the timed window (mark_start / mark_end)."""
    Q = ("clocks.sm,clocks.max.sm,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []  # (host time, fields)
        self.proc = None
        self.t0 = self.t1 = None
        self.first = threading.Event()

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None
        return self

    def wait_first(self, timeout: float = 5.0) -> bool:
        """Block until the first sample has arrived (nvidia-smi takes a few
        hundred ms to start), so that a short timed region is still sampled."""
        return self.proc is not None and self.first.wait(timeout)

    def mark_start(self):
        self.t0 = time.monotonic()

    def mark_end(self):
        self.t1 = time.monotonic()

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) == 6:
                self.rows.append((time.monotonic(), parts))
                self.first.set()

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def window(self):
        """The samples of the timed window; if it was shorter than the sampling
        period, the sample nearest to its middle."""
        if not self.rows:
            return []
        t0 = self.t0 if self.t0 is not None else -1e300
        t1 = self.t1 if self.t1 is not None else 1e300
        inside = [r for t, r in self.rows if t0 <= t <= t1]
        if inside:
            return inside
        mid = 0.5 * (t0 + t1) if self.t0 is not None and self.t1 is not None else t1
        return [min(self.rows, key=lambda tr: abs(tr[0] - mid))[1]]

    def summary(self):
        rows = self.window()
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = sorted(float(r[0]) for r in rows if r[0].replace(".", "").isdigit())
        mx = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4)
                          if r[2 + i].lower() == "active"})
        return {"sm_mhz": sm[len(sm) // 2] if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows), "samples_total": len(self.rows)}


# the timed region is repeated until it has lasted at least this long
MIN_TIMED_SECONDS = 1.0
# warm-up steps beyond the requested ones: enough to capture the step graph
# (64 steps), let a batch time its tile shapes and bring the clocks up
MIN_WARMUP_STEPS = 192


def timed_blocks(step, k: int, stream, min_seconds: float = MIN_TIMED_SECONDS,
                 max_blocks: int = 100000):
    """Run step(k) R times back to back, each bracketed by CUDA events on the
    launching stream, until the blocks have taken at least min_seconds of
    device time; returns the per-block device times in ms.  The first block is
    timed alone to size R, so that the whole region is queued without host
    synchronisation between blocks."""
    import torch
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    step(k)
    e1.record(stream)
    torch.cuda.synchronize()
    times = [e0.elapsed_time(e1)]
    need = int(min(max_blocks, max(0, min_seconds * 1e3 / max(times[0], 1e-3) - 1)))
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(need)]
    for a, b in evs:
        a.record(stream)
        step(k)
        b.record(stream)
    torch.cuda.synchronize()
    times += [a.elapsed_time(b) for a, b in evs]
    return times


def median(v):
    s = sorted(v)
    n = len(s)
    return s[n // 2] if n % 2 else 0.5 * (s[n // 2 - 1] + s[n // 2])


def channel_sample(nx, ny, tau_f=0.6, w0=2.0, u0=0.35, radius=11.0, umax=0.005):
    """Inputs of one closed-channel problem (the centre of the c5 sweep):
    tanh seed at the centre, uniform U0, Poiseuille profile of a body force."""
    import numpy as np
    nu = (tau_f - 0.5) / 3.0
    g = 8.0 * nu * umax / (ny * ny)
    y, x = np.mgrid[0:ny, 0:nx].astype(np.float64)
    phi = np.tanh((radius - np.hypot(x - nx // 2, y - ny // 2)) / (np.sqrt(2.0) * w0))
    ux = g / (2.0 * nu) * (y + 0.5) * (ny - 0.5 - y)
    return g, dict(phi=phi, U=np.full_like(phi, u0), ux=ux, uy=np.zeros_like(phi))


def oracle_problem(w):
    import oracle
    s = w["sample"]
    body = (0.0, 0.0, 0.0)
    if s.get("channel"):
        g, f = channel_sample(s["nx"], s["ny"])
        body = (g, 0.0, 0.0)
    p = oracle.Params(dim=w["dim"], nx=s["nx"], ny=s["ny"], nz=s.get("nz", 1), bc=w["bc"],
                      flow=w["flow"], fold=w["fold"], eps=w["eps"], u_inlet=w["u_in"],
                      u0_inlet=w["U_in"], body=body, theta0=w.get("theta0", 0.0),
                      collision=w.get("collision", 0))
    o = oracle.Oracle(p)
    if s.get("channel"):
        o.init_fields(f["phi"], f["U"], None, f["ux"], f["uy"])
    elif s.get("polygon"):
        g = s["polygon"]
        nrm, d = hexagon(g["perimeter"], w["theta0"] + 3.141592653589793 / 6)
        o.init_polygon(g["cx"], g["cy"], nrm, d, g["u0"], g["noise"], g["seed"])
    else:
        o.init_seed(*s["seed"])
    if s.get("baffle"):
        o.set_solid(baffle_mask(s["nx"], s["ny"], s["baffle"]))
    return p, o


def hexagon(perimeter, theta):
    """Side normals (counter-clockwise from theta) and apothems of a regular
    hexagon of the given perimeter."""
    import numpy as np
    a = theta + np.pi / 3.0 * np.arange(6)
    return np.stack([np.cos(a), np.sin(a)], axis=1), np.full(6, perimeter / 6.0 * 3 ** 0.5 / 2)


def baffle_mask(nx, ny, b):
    """Solid mask [ny, nx] with a baffle of b["w"] columns at b["x0"], rows
    b["y0"] .. b["y1"] - 1."""
    import numpy as np
    m = np.zeros((ny, nx), np.uint8)
    m[b["y0"]:b["y1"], b["x0"]:b["x0"] + b["w"]] = 1
    return m


def oracle_sample(w, seconds: float, threads: int):
    """The FP64 CPU oracle, as it stands, on a bounded sample of the workload."""
    p, o = oracle_problem(w)
    o.step(1, threads)
    steps, t0 = 0, time.perf_counter()
    while time.perf_counter() - t0 < seconds:
        o.step(1, threads)
        steps += 1
    dt = time.perf_counter() - t0
    return p.nodes * steps / dt / 1e6, steps, p.nodes, dt


def run_reference(args, w):
    """The oracle on the host cores: each step advances a bounded sample."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    threads = os.cpu_count() or 1
    s = w["sample"]
    p, o = oracle_problem(w)
    if w.get("surrogate"):  # LB-equivalent steps: the oracle runs the LB
        args.steps = min(args.steps, 200)
    for _ in range(args.warmup):
        o.step(1, threads)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        o.step(1, threads)
    dt = time.perf_counter() - t0
    v = p.nodes * args.steps / dt / 1e6
    sample = (f"{s['nx']}x{s['ny']}" + (f"x{s['nz']}" if w['dim'] == 3 else "") +
              " nodes of the same workload per step (FP64 oracle, OpenMP)")
    metric = ("LB-equivalent MLUPS (learned block propagator)" if w.get("surrogate")
              else "coupled-LB MLUPS")
    print(json.dumps({
        "impl": "reference", "metric": metric, "value": v, "unit": "MLUPS",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": dt / args.steps * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w["desc"], "sample_grid": [s["nx"], s["ny"], s.get("nz", 1)]},
        "cpu_baseline": {"value": v, "unit": "MLUPS", "cores": threads, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": v, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20000)
    ap.add_argument("--warmup", type=int, default=200)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="c2", choices=sorted(WORKLOADS))
    ap.add_argument("--e2e-steps", type=int, default=50)
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    w = workload(args.workload, int(os.environ.get("RANK", "0")),
                 int(os.environ.get("WORLD_SIZE", "1")))
    if args.impl == "reference":
        return run_reference(args, w)
    if w.get("surrogate"):
        return run_surrogate(args, w)
    if w.get("network"):
        return run_network(args, w)
    if w.get("polygon"):
        return run_facets(args, w)

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

    def barrier():
        if dist is not None:
            dist.barrier()

    import paper_2206_02145_gb300 as L
    stream = torch.cuda.current_stream()
    batch = None
    if w.get("batch"):
        params, seeds = w["members"]
        st = lib_params(w, L)["storage"]
        batch = L.Batch([dict(p, storage=st) for p in params], seeds, stream.cuda_stream)
        sims = [batch.instance(i) for i in range(batch.count)]
        stepper = batch
    else:
        sim = L.Sim(stream=stream.cuda_stream, **lib_params(w, L))
        if w.get("baffle"):
            sim.set_solid(baffle_mask(w["nx"], w["ny"], w["baffle"]))
        sim.init_seed(*w["seed"])
        sims = [sim]
        stepper = sim

    # interface rays of the initial state (for the growth comparison below)
    d_init = [s_.diagnostics()["iface_pos"] for s_ in sims]

    with ClockSampler(local) as clk:
        clk.wait_first()
        # warm-up: at least MIN_WARMUP_STEPS, so that the step graph is built
        # (and a batch has timed its tile shapes) before the timed region
        warm = max(args.warmup, MIN_WARMUP_STEPS)
        stepper.step(warm)
        torch.cuda.synchronize()

        # --- device-resident timed region: R blocks of K steps, inputs in HBM ---
        barrier()
        torch.cuda.synchronize()
        clk.mark_start()
        blocks = timed_blocks(stepper.step, args.steps, stream)
        clk.mark_end()
        barrier()
    reps = len(blocks)
    ms = median(blocks)  # median device time of one block of K steps
    ms_max = max_over_ranks([ms], dist)[0]
    per_step_ms = ms_max / args.steps
    value = w["nodes_all"] * args.steps / (ms_max * 1e-3) / 1e6
    diags = [s.diagnostics() for s in sims]  # also surfaces any sticky device error
    d = diags[0]
    total_steps = warm + args.steps * reps

    def same_steps_plain(storage=None, collision=None):
        """The same problem in another storage or collision, brought through the
        same warm-up and timed blocks; returns its median block time (ms) and
        its final interface rays."""
        kw = lib_params(w, L, storage=storage)
        if collision is not None:
            kw["collision"] = collision
        q = L.Sim(stream=stream.cuda_stream, **kw)
        if w.get("baffle"):
            q.set_solid(baffle_mask(w["nx"], w["ny"], w["baffle"]))
        q.init_seed(*w["seed"])
        q.step(warm)
        torch.cuda.synchronize()
        t = timed_blocks(q.step, args.steps, stream, max_blocks=reps - 1)
        left = total_steps - warm - args.steps * len(t)
        if left > 0:
            q.step(left)
        iface = q.diagnostics()["iface_pos"]
        q.close()
        return max_over_ranks([median(t)], dist)[0], iface

    vs_fp32 = None
    if batch is None and w["storage"] != "fp32":
        # the plain form: the same problem in FP32 storage, the same steps
        ms32, iface32 = same_steps_plain(storage="fp32")
        e, rel = iface_compare(d_init[0], d["iface_pos"], iface32, w["dim"])
        vs_fp32 = {"plain_fp32_ms_per_step": ms32 / args.steps,
                   "speedup": ms32 / ms_max, "steps": total_steps,
                   "iface_pos_err_lu": e, "growth_rel_err": rel}

    fp16_form = None
    if batch is None and w["storage"] == "fp32" and w.get("fp16_compare"):
        # the FP16-storage form of the same problem over the same steps: its
        # speed-up over this FP32 run and its interface against it
        ms16, iface16 = same_steps_plain(storage="fp16")
        e, rel = iface_compare(d_init[0], iface16, d["iface_pos"], w["dim"])
        fp16_form = {"fp16_ms_per_step": ms16 / args.steps, "speedup_over_fp32": ms_max / ms16,
                     "steps": total_steps, "iface_pos_err_lu": e, "growth_rel_err": rel}
        # its own HBM roofline: algorithmic bytes of the FP16 node update over
        # the same measured copy peak as the FP32 line
        b16 = lup_bytes(w, "fp16")
        gbs16 = b16 * w["nodes"] / (ms16 / args.steps * 1e-3) / 1e9
        fp16_form.update({"bytes_per_lup": b16, "achieved_gbs": gbs16,
                          "hbm_frac": gbs16 / measured_peaks()[0]})

    vs_bgk = None
    if batch is None and w.get("collision"):
        # the same problem with the BGK collision (Eq. 8), the same steps
        msb, ifaceb = same_steps_plain(collision=0)
        e, rel = iface_compare(d_init[0], d["iface_pos"], ifaceb, w["dim"])
        vs_bgk = {"bgk_ms_per_step": msb / args.steps, "time_ratio_chm_over_bgk": ms_max / msb,
                  "steps": total_steps, "iface_pos_diff_lu": e, "growth_rel_diff": rel}

    batch_info = None
    if batch is not None:
        # the same instances stepped one after another (each its own graph),
        # against the single batched launch per step
        kseq = max(64, min(args.steps, 640) // 64 * 64)
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for s_ in sims:
            s_.step(64)
        torch.cuda.synchronize()
        ev0.record(stream)
        for s_ in sims:
            s_.step(kseq)
        ev1.record(stream)
        torch.cuda.synchronize()
        seq_ms = ev0.elapsed_time(ev1) / kseq
        # the plain form: the same instances in FP32 storage, one after another
        params32, seeds32 = w["members"]
        plain = []
        for p_, s_ in zip(params32, seeds32):
            q = L.Sim(stream=stream.cuda_stream, **dict(p_, storage=L.FP32))
            q.init_seed(*s_)
            plain.append(q)
        for q in plain:
            q.step(64)
        torch.cuda.synchronize()
        ev0.record(stream)
        for q in plain:
            q.step(kseq)
        ev1.record(stream)
        torch.cuda.synchronize()
        fp32_ms = ev0.elapsed_time(ev1) / kseq
        # accuracy: every plain FP32 instance brought to the batch's step count
        left = total_steps - 64 - kseq
        for q in plain:
            if left > 0:
                q.step(left)
        errs, rels = [], []
        for i, q in enumerate(plain):
            e, rel = iface_compare(d_init[i], diags[i]["iface_pos"],
                                   q.diagnostics()["iface_pos"], 2)
            if e is not None:
                errs.append(e)
            rels.extend(rel)
            q.close()
        batch_info = {"instances": batch.count, "tuning": batch.tuning(),
                      "sequential_ms_per_step": seq_ms,
                      "speedup_vs_sequential": seq_ms / per_step_ms,
                      "plain_fp32_sequential_ms_per_step": fp32_ms,
                      "speedup_vs_plain_fp32": fp32_ms / per_step_ms,
                      "vs_plain_fp32_after_steps": total_steps,
                      "iface_pos_err_lu_max": max(errs) if errs else None,
                      "growth_rel_err_max": max((abs(r) for r in rels), default=None),
                      "growth_rel_err_median": (sorted(abs(r) for r in rels)[len(rels) // 2]
                                                if rels else None)}

    # --- end to end through the C ABI with host buffers -------------------------
    # every step: H2D of the full state from pinned memory (lbpf_write_state),
    # one coupled step, D2H of phi and U (lbpf_read_fields); for a batch, of
    # every instance
    host_states = [torch.from_numpy(s_.state()).pin_memory() for s_ in sims]
    nf = 2
    host_outs = [torch.empty(nf * s_.nodes, dtype=torch.float32).pin_memory() for s_ in sims]
    mask = L.FIELD_PHI | L.FIELD_U

    def e2e_step():
        for s_, hs_ in zip(sims, host_states):
            L.lbpf_write_state(s_.h, hs_.data_ptr(), hs_.numel())
        stepper.step(1)
        for s_, ho_ in zip(sims, host_outs):
            L.lbpf_read_fields(s_.h, mask, ho_.data_ptr(), ho_.numel() * 4, 0)

    for _ in range(3):
        e2e_step()
    barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.e2e_steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    e2e_max = max_over_ranks([e2e_s], dist)[0]
    e2e_value = w["nodes_all"] * args.e2e_steps / e2e_max / 1e6
    h2d = sum(int(x.numel()) for x in host_states)
    d2h = sum(int(x.numel()) * 4 for x in host_outs)

    peak, peak_kind = measured_peaks()
    achieved = w["bytes_per_lup"] * w["nodes"] / (per_step_ms * 1e-3) / 1e9
    traffic = profiled_traffic(w)
    clocks = clk.summary()
    if clocks.get("sm_mhz"):
        # the step time scaled to the median SM clock seen (ms x MHz): compares
        # runs taken at different clocks
        clocks["ms_per_step_x_mhz"] = per_step_ms * clocks["sm_mhz"]

    if rank == 0:
        cpu = None
        if not args.no_cpu_baseline:
            threads = os.cpu_count() or 1
            v, steps, n, dt = oracle_sample(w, args.cpu_seconds, threads)
            s = w["sample"]
            cpu = {"value": v, "unit": "MLUPS", "cores": threads, "kind": "oracle",
                   "sample": f"{steps} steps of a {s['nx']}x{s['ny']}"
                             + (f"x{s['nz']}" if w['dim'] == 3 else "")
                             + f" grid of the same workload ({n} nodes), {dt:.1f} s, FP64"}
        out = {
            "metric": "coupled-LB MLUPS", "value": value, "unit": "MLUPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": per_step_ms,
            "timing": {"blocks": reps, "steps_per_block": args.steps,
                       "statistic": "median over blocks (CUDA events on the step stream)",
                       "ms_per_block_median": ms, "ms_per_block_mean": sum(blocks) / reps,
                       "ms_per_block_min": min(blocks), "ms_per_block_max": max(blocks),
                       "timed_s": sum(blocks) * 1e-3, "warmup_steps_run": warm},
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32" if w["storage"] == "fp32" else (
                "f64" if w["storage"] == "fp64" else f"f32 ({w['storage']} storage)"),
            "data": "synthetic (seeded tanh seed + SplitMix64 noise)",
            "config": {"workload": w["desc"], "grid": [w["nx"], w["ny"], w["nz"]],
                       "storage": w["storage"], "bytes_per_lup": w["bytes_per_lup"],
                       "l2": f"inputs larger than L2: {w['bytes_per_lup'] * w['nodes'] / 1e6:.0f}"
                             " MB moved per step vs 129 MB L2",
                       "parallelism": "single GPU" if world == 1 else (
                           f"sweep of {w['batch'] * world} instances sharded over {world} GPUs"
                           if w.get("batch") else "replicas")},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "peak_source": peak_kind,
                         "frac_of_nominal_7900": achieved / 7900.0,
                         "traffic": traffic,
                         "algorithmic_bytes_per_launch": w["bytes_per_lup"] * w["nodes"]},
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": "MLUPS",
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
            "gpu_launches": args.steps * reps,
            "clocks": clocks,
            "diag": {"step": d["step"], "solute_drift_rel": d["solute_drift_rel"],
                     "r_eq": d["r_eq"]},
        }
        if vs_fp32 is not None:
            out["vs_plain_fp32"] = vs_fp32
        if fp16_form is not None:
            out["fp16_storage"] = fp16_form
        if vs_bgk is not None:
            out["vs_bgk"] = vs_bgk
        if batch_info is not None:
            out["config"]["batch"] = batch_info
            out["config"]["grid"] = "64 square grids, sides 256..768"
        print(json.dumps(out), flush=True)
    del sims
    stepper.close()
    if dist is not None:
        dist.destroy_process_group()


def run_facets(args, w):
    """f1: the coupled step with the crystal-shape measurement every `every`
    steps (one GPU; replicas beyond).  value = MLUPS of the whole run,
    measurements included; beside it the measurement's own time and HBM
    roofline, and the growth-rate fits of the side lengths."""
    import numpy as np
    import torch
    import paper_2206_02145_gb300 as L
    local = int(os.environ.get("LOCAL_RANK", "0"))
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    stream = torch.cuda.current_stream()
    g = w["polygon"]
    nrm, dist0 = hexagon(g["perimeter"], w["theta0"] + np.pi / 6)
    sim = L.Sim(stream=stream.cuda_stream, **lib_params(w, L))
    sim.init_polygon(g["cx"], g["cy"], nrm, dist0, g["u0"], g["noise"], g["seed"])
    every = w["every"]
    steps = max(every, args.steps // every * every)
    sim.step(args.warmup)
    first = sim.facets(nrm)
    torch.cuda.synchronize()
    hist_t, hist_L = [args.warmup], [first["L"]]
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        clk.wait_first()
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()
        clk.mark_start()
        ev0.record(stream)
        for k in range(steps // every):
            sim.step(every)
            r = sim.facets(nrm)
            hist_t.append(args.warmup + (k + 1) * every)
            hist_L.append(r["L"])
        ev1.record(stream)
        torch.cuda.synchronize()
        clk.mark_end()
        if dist is not None:
            dist.barrier()
    ms = max_over_ranks([ev0.elapsed_time(ev1)], dist)[0]
    value = whole_job_rate(w["nodes"] * steps, world, ms * 1e-3) / 1e6
    # the measurement alone: blocking calls (host round trip included), and
    # the device part queued back to back (support pass, final reduction, the
    # copy of 21 numbers; an upper bound of the device time where the host's
    # launches are the slower side)
    nrep = 50
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(nrep):
        sim.facets(nrm)
    call_us = (time.perf_counter() - t0) / nrep * 1e6
    torch.cuda.synchronize()
    ev0.record(stream)
    for _ in range(nrep):
        L.lbpf_facets_enqueue(sim.h, nrm)
    ev1.record(stream)
    torch.cuda.synchronize()
    meas_us = ev0.elapsed_time(ev1) / nrep * 1e3
    L.lbpf_facets_collect(sim.h)
    # algorithmic bytes of one measurement: the 9 h populations of every node
    # read once (FP32)
    meas_bytes = 9 * 4 * w["nodes"]
    peak, peak_kind = measured_peaks()
    ach = meas_bytes / (meas_us * 1e-6) / 1e9
    Lh = np.array(hist_L)
    t = np.array(hist_t, dtype=np.float64)
    fits = [L.lbpf_growth_fit(t, Lh[:, i]) for i in range(Lh.shape[1])]
    favg = L.lbpf_growth_fit(t, Lh.mean(axis=1))
    d = sim.diagnostics()
    if rank == 0:
        cpu = None
        if not args.no_cpu_baseline:
            threads = os.cpu_count() or 1
            v, st, n, dt = oracle_sample(w, args.cpu_seconds, threads)
            cpu = {"value": v, "unit": "MLUPS", "cores": threads, "kind": "oracle",
                   "sample": f"{st} LB steps of a 256x256 grid of the same workload ({n} "
                             f"nodes), {dt:.1f} s, FP64"}
        print(json.dumps({
            "metric": "coupled-LB MLUPS (with crystal-shape measurement)", "value": value,
            "unit": "MLUPS", "n_gpus": world, "steps": steps, "warmup": args.warmup,
            "ms_per_step": ms / steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic (seeded hexagonal seed + "
            "SplitMix64 noise)",
            "config": {"workload": w["desc"], "grid": [w["nx"], w["ny"], 1], "every": every,
                       "l2": "inputs larger than L2: 235 MB moved per step vs 129 MB L2",
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "shape": {"L_initial": first["L"].tolist(), "L_final": hist_L[-1].tolist(),
                      "growth_rate_lu_per_step": [f[0] for f in fits],
                      "r2": [f[2] for f in fits],
                      "L_avg_growth_rate": favg[0], "L_avg_r2": favg[2],
                      "Q": float(Lh[-1].max() / Lh[-1].min()), "aspect": r["aspect"],
                      "centre": r["centre"].tolist(), "samples": len(hist_t)},
            "measurement": {"us_per_call": call_us, "device_us": meas_us, "share_of_run":
                            (steps // every) * call_us * 1e-3 / ms},
            "roofline": {"bound": "hbm",
                         "kernel": "facet_support_kernel (+ result reset and copy)",
                         "achieved": ach, "peak": peak, "unit": "GB/s", "frac": ach / peak,
                         "peak_source": peak_kind,
                         "traffic": profiled_traffic(dict(kernel="facet_support_kernel",
                                                          nx=w["nx"], storage="fp32",
                                                          src=SRC_FACETS)),
                         "algorithmic_bytes_per_launch": meas_bytes},
            "cpu_baseline": cpu,
            "gpu_launches": steps + (steps // every),  # the step, one shape kernel each
            "clocks": clk.summary(),
            "diag": {"step": d["step"], "solute_drift_rel": d["solute_drift_rel"]},
        }), flush=True)
    sim.close()
    if dist is not None:
        dist.destroy_process_group()


def unet_forward_flops(nx, ny, batch=1):
    """Algorithmic FLOPs of one forward pass of the 4-level 32/64/128/256 U-Net
    (3x3 convolutions only; 2 flops per multiply-add)."""
    Cs = [32, 64, 128, 256]
    flop = 0
    for lev in range(4):
        px = batch * (ny >> lev) * (nx >> lev)
        flop += 2 * 9 * px * ((16 if lev == 0 else Cs[lev - 1]) * Cs[lev] + Cs[lev] * Cs[lev])
        if lev < 3:
            flop += 2 * 9 * px * (Cs[lev + 1] * Cs[lev] + 3 * Cs[lev] * Cs[lev])
    return flop


def run_network(args, w):
    """c5net: the network's kernels alone, K forward passes then K training steps."""
    import torch
    import paper_2206_02145_gb300 as L
    B = w["network"]["batch"]
    nx, ny = w["nx"], w["ny"]
    stream = torch.cuda.current_stream()
    net = L.UNet(in_ch=4, out_ch=4, levels=4, batch=B, height=ny, width=nx, seed=1,
                 stream=stream.cuda_stream)
    g = torch.Generator(device="cpu").manual_seed(0)
    x = torch.randn(B, ny, nx, 4, generator=g).cuda()
    t = torch.randn(B, ny, nx, 4, generator=g).cuda()
    y = torch.empty_like(x)
    for _ in range(args.warmup):
        net.forward(x, y)
        net.train_step(x, t, 1e-5)
    # one forward pass and one training step inside NVTX ranges ("forward",
    # "train_step"), so that a profiler can capture exactly their launches
    # (ncu --nvtx --nvtx-include forward/)
    torch.cuda.nvtx.range_push("forward")
    net.forward(x, y)
    torch.cuda.nvtx.range_pop()
    torch.cuda.nvtx.range_push("train_step")
    net.train_step(x, t, 1e-5)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    with ClockSampler(int(os.environ.get("LOCAL_RANK", "0"))) as clk:
        clk.wait_first()
        clk.mark_start()
        ev[0].record(stream)
        for _ in range(args.steps):
            net.forward(x, y)
        ev[1].record(stream)
        for _ in range(args.steps):
            net.train_step(x, t, 1e-5)
        ev[2].record(stream)
        torch.cuda.synchronize()
        clk.mark_end()
    net.status()
    fwd = ev[0].elapsed_time(ev[1]) / args.steps
    trn = ev[1].elapsed_time(ev[2]) / args.steps
    flop = unet_forward_flops(nx, ny, B)
    tf = flop / (fwd * 1e-3) / 1e12
    peak_tf, peak_kind = measured_bf16()
    print(json.dumps({
        "metric": "U-Net forward TFLOP/s", "value": tf, "unit": "TFLOP/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": fwd,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
        "data": "synthetic (random weights and inputs)",
        "config": {"workload": w["desc"], "batch": B, "params": net.param_count},
        "train_step_ms": trn, "train_tflops": 3 * flop / (trn * 1e-3) / 1e12,
        "roofline": {"bound": "tensor", "achieved": tf, "peak": peak_tf, "unit": "TFLOP/s",
                     "frac": tf / peak_tf, "peak_source": peak_kind, "traffic": None},
        "clocks": clk.summary()}), flush=True)
    net.close()


def surrogate_arm(args, w, nb, stream, dist, clk, rank):
    """Train the network for blocks of nb LB steps (pairs from the LB, training
    on the GPU) and time the block propagator against the plain LB over the
    same LB-equivalent steps of a held-out problem.  Returns the arm's figures
    and its inference network (closed by the caller)."""
    import numpy as np
    import torch
    import paper_2206_02145_gb300 as L
    from paper_2206_02145_gb300 import surrogate as S
    c = w["surrogate"]
    nx, ny = w["nx"], w["ny"]
    cfg = S.default_cfg(nb)
    t0 = time.perf_counter()
    # pairs every `every` steps along each trajectory, the block nb apart
    X, T = S.generate_pairs(c["traj"], c["t_end"], c["every"], nx, ny, cfg, seed=100,
                            crop=c["crop"])
    t_data = time.perf_counter() - t0
    train_steps, lr = c["recipe"][nb]
    # validation (a problem of its own, neither a training trajectory nor the
    # held-out test problem): the network alone advances val_steps LB steps
    # worth of blocks (only the first is judged) and its interface is compared
    # with the LB's; a candidate that drifts by more than val_tol lattice units
    # is replaced by one trained from the next initialisation seed (at most
    # val_seeds); the best candidate is kept
    vblocks = max(4, c["val_steps"] // nb)
    vparams, vfields, _ = S.channel_problem(np.random.default_rng(5151 + rank), nx, ny)
    vb = S.make_sim(vparams, vfields, stream.cuda_stream)
    vb.step(c["start"] + vblocks * nb)
    v_ref = vb.diagnostics()["iface_pos"][:4]
    vb.close()
    vcfg = S.default_cfg(nb, judge_every=0, drift_tol=1.0, iface_tol=1e9)
    t0 = time.perf_counter()
    tries = []
    tr = None
    for nseed in range(1, c["val_seeds"] + 1):
        cand = L.UNet(in_ch=4, out_ch=4, levels=4, batch=c["batch"], height=c["crop"],
                      width=nx, seed=nseed, stream=stream.cuda_stream)
        h_ = S.train(cand, X, T, train_steps, lr=lr, log_every=1000)
        cand.status()
        vnet = S.inference_net(cand, nx, ny, stream.cuda_stream)
        va = S.make_sim(vparams, vfields, stream.cuda_stream)
        va.step(c["start"])
        L.lbpf_surrogate_advance(va, vnet, vcfg, vblocks)
        verr = float(np.max(np.abs(va.diagnostics()["iface_pos"][:4] - v_ref)))
        va.close()
        vnet.close()
        tries.append({"seed": nseed, "val_iface_err_lu": verr})
        if tr is None or verr < best:
            if tr is not None:
                tr.close()
            tr, hist, best = cand, h_, verr
        else:
            cand.close()
        if verr <= c["val_tol"]:
            break
    t_train = time.perf_counter() - t0
    npairs = int(X.shape[0])
    del X, T
    # held-out pairs (other problems): the network's error against predicting no change
    Xv, Tv = S.generate_pairs(3, c["t_end"], 2 * c["every"], nx, ny, cfg, seed=999,
                              crop=c["crop"])
    ev = S.inference_net(tr, nx, c["crop"], stream.cuda_stream)
    mse_net, mse_none = S.prediction_error(ev, Xv, Tv)
    ev.close()
    del Xv, Tv
    net = S.inference_net(tr, nx, ny, stream.cuda_stream)
    tr.close()

    # held-out problem: propagator (a) and plain LB (b) from the same state
    rng = np.random.default_rng(4242 + rank)
    params, fields, info = S.channel_problem(rng, nx, ny)
    a = S.make_sim(params, fields, stream.cuda_stream)
    b = S.make_sim(params, fields, stream.cuda_stream)
    a.step(c["start"])
    b.step(c["start"])
    pcfg = S.default_cfg(nb, judge_every=c["judge_every"], drift_tol=1e-3, iface_tol=1.0,
                         iface_rel_tol=c["iface_rel_tol"])
    L.lbpf_surrogate_advance(a, net, pcfg, 1)  # warm-up: captures the prediction graph
    b.step(nb)
    torch.cuda.synchronize()
    d0 = b.diagnostics()
    # --steps is a minimum: the comparison spans at least c["min_steps"] LB steps,
    # so that the judged blocks (one in judge_every) weigh as they do in a run
    K = max(1, max(args.steps, c["min_steps"]) // nb)
    steps = K * nb
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    clk.mark_start()
    ev0.record(stream)
    rep = L.lbpf_surrogate_advance(a, net, pcfg, K)
    ev1.record(stream)
    torch.cuda.synchronize()
    ms_s = ev0.elapsed_time(ev1)
    ev0.record(stream)
    b.step(steps)
    ev1.record(stream)
    torch.cuda.synchronize()
    clk.mark_end()
    ms_lb = ev0.elapsed_time(ev1)
    ms_s, ms_lb = max_over_ranks([ms_s, ms_lb], dist)
    da, db = a.diagnostics(), b.diagnostics()
    grow_lb = db["iface_pos"][:4] - d0["iface_pos"][:4]
    grow_s = da["iface_pos"][:4] - d0["iface_pos"][:4]
    rel = (grow_s - grow_lb) / np.where(np.abs(grow_lb) > 1e-9, np.abs(grow_lb), np.nan)

    # the same held-out run with the accumulated interface estimate bounded at
    # 1 lattice unit (the controller then hands the rest of the run to the LB)
    cb = S.make_sim(params, fields, stream.cuda_stream)
    cb.step(c["start"] + nb)
    bcfg = S.default_cfg(nb, judge_every=c["judge_every"], drift_tol=1e-3, iface_tol=1.0,
                         iface_rel_tol=c["iface_rel_tol"], iface_budget=1.0)
    torch.cuda.synchronize()
    ev0.record(stream)
    rep_b = L.lbpf_surrogate_advance(cb, net, bcfg, K)
    ev1.record(stream)
    torch.cuda.synchronize()
    ms_b = ev0.elapsed_time(ev1)
    dcb = cb.diagnostics()
    grow_b = dcb["iface_pos"][:4] - d0["iface_pos"][:4]
    budgeted = {"iface_budget_lu": 1.0, "speedup_vs_plain_lb": ms_lb / ms_b, "report": rep_b,
                "growth_lu": grow_b.tolist(),
                "iface_pos_error_lu": float(np.max(np.abs(dcb["iface_pos"][:4] -
                                                          db["iface_pos"][:4])))}
    cb.close()
    b.close()
    nodes = nx * ny * w.get("world", 1)
    return {
        "block_steps": nb, "steps": steps, "blocks": K, "ms": ms_s, "plain_lb_ms": ms_lb,
        "value": nodes * steps / (ms_s * 1e-3) / 1e6,
        "plain_lb_value": nodes * steps / (ms_lb * 1e-3) / 1e6,
        "speedup_vs_plain_lb": ms_lb / ms_s, "report": rep,
        "growth_lu": {"plain_lb": grow_lb.tolist(), "propagator": grow_s.tolist(),
                      "rel_error": [None if not np.isfinite(x) else float(x) for x in rel]},
        "growth_rel_err_max": float(np.nanmax(np.abs(rel))) if np.isfinite(rel).any() else None,
        "iface_pos_error_lu": float(np.max(np.abs(da["iface_pos"][:4] - db["iface_pos"][:4]))),
        "solute_drift_rel": da["solute_drift_rel"],
        "with_accumulated_bound": budgeted,
        "training": {"pairs": npairs, "steps": train_steps, "lr": lr, "batch": c["batch"],
                     "band_rows": c["crop"], "data_s": round(t_data, 1),
                     "train_s": round(t_train, 1), "loss": [round(x[1], 5) for x in hist],
                     "validation": {"blocks": vblocks, "tol_lu": c["val_tol"],
                                    "candidates": tries},
                     "held_out_mse": mse_net, "held_out_mse_no_network": mse_none,
                     "held_out_ratio": mse_net / mse_none},
        "held_out_problem": info,
    }, net, a, pcfg, K


def propagator_launches(rep, nb):
    """Kernels of one lbpf_surrogate_advance on the configured network, from its
    report: every block's prediction (read-out 2, network 19, predicted planes 1,
    their sums 2 and interface positions 1), two to commit a predicted block, nb
    steps for the others (the two of the last read-out, where the last block was
    the LB's, are not counted)."""
    lb = rep["judged_blocks"] + rep["fallback_blocks"]
    return rep["blocks"] * 25 + rep["surrogate_blocks"] * 2 + lb * nb


def run_surrogate(args, w):
    """c5: for each block length (the configured 50 LB steps first, then 200),
    train the U-Net on LB trajectories and time the block propagator against
    the plain LB on a held-out problem (one GPU; replicas beyond).  The line's
    value is the configured block's; the other is reported beside it."""
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
    import paper_2206_02145_gb300 as L
    c = w["surrogate"]
    nx, ny = w["nx"], w["ny"]
    w = dict(w, world=world)
    stream = torch.cuda.current_stream()
    arms, keep = {}, None
    with ClockSampler(local) as clk:
        clk.wait_first()
        for nb in c["blocks"]:
            res, net, a, pcfg, K = surrogate_arm(args, w, nb, stream, dist, clk, rank)
            arms[nb] = res
            if keep is None:
                keep = (net, a, pcfg, K, nb)
            else:
                net.close()
                a.close()
    net, a, pcfg, K, nb = keep
    head = arms[nb]

    # the network forward alone: the tensor-core part of the path
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    xs = torch.zeros(ny, nx, 4, device="cuda")
    ys = torch.empty_like(xs)
    for _ in range(3):
        net.forward(xs, ys)
    torch.cuda.synchronize()
    ev0.record(stream)
    for _ in range(20):
        net.forward(xs, ys)
    ev1.record(stream)
    torch.cuda.synchronize()
    fwd_ms = ev0.elapsed_time(ev1) / 20
    flop = unet_forward_flops(nx, ny)
    tflops = flop / (fwd_ms * 1e-3) / 1e12
    peak_tf, peak_kind = measured_bf16()

    # --- end to end through the C ABI with host buffers ---------------------------
    # per call: the state from pinned host memory (lbpf_write_state), Ke blocks
    # of the propagator, phi and U back to pinned host memory
    nodes = nx * ny
    hs = torch.from_numpy(a.state()).pin_memory()
    ho = torch.empty(2 * nodes, dtype=torch.float32).pin_memory()
    Ke = min(K, 10)
    L.lbpf_write_state(a.h, hs.data_ptr(), hs.numel())
    L.lbpf_surrogate_advance(a, net, pcfg, 1)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    L.lbpf_write_state(a.h, hs.data_ptr(), hs.numel())
    L.lbpf_surrogate_advance(a, net, pcfg, Ke)
    L.lbpf_read_fields(a.h, L.FIELD_PHI | L.FIELD_U, ho.data_ptr(), ho.numel() * 4, 0)
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    e2e_value = nodes * world * Ke * nb / e2e_s / 1e6

    if rank == 0:
        cpu = None
        if not args.no_cpu_baseline:
            threads = os.cpu_count() or 1
            v, osteps, n, dt = oracle_sample(w, args.cpu_seconds, threads)
            cpu = {"value": v, "unit": "MLUPS", "cores": threads, "kind": "oracle",
                   "sample": f"{osteps} LB steps of a 256x256 closed channel of the same family "
                             f"({n} nodes), {dt:.1f} s, FP64"}
        rep = head["report"]
        launches = propagator_launches(rep, nb)
        out = {
            "metric": "LB-equivalent MLUPS (learned block propagator)", "value": head["value"],
            "unit": "MLUPS", "n_gpus": world, "steps": head["steps"], "warmup": nb,
            "ms_per_step": head["ms"] / head["steps"], "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "bf16 network, f32 LB",
            "data": "synthetic (seeded channel problems; the network's training pairs come "
                    "from this LB)",
            "config": {"workload": w["desc"], "grid": [nx, ny, 1], "block_steps": nb,
                       "judge_every": c["judge_every"], "training": head["training"],
                       "held_out_problem": head["held_out_problem"],
                       "l2": "network activations of a 512x512 sample exceed L2 at level 0 "
                             "only partly; the LB state (59 MB) fits in L2: both arms time the "
                             "same K blocks back to back",
                       "parallelism": "replicas" if world > 1 else "single GPU"},
            "plain_lb": {"value": head["plain_lb_value"], "unit": "MLUPS",
                         "ms": head["plain_lb_ms"]},
            "speedup_vs_plain_lb": head["speedup_vs_plain_lb"],
            "report": rep,
            "growth_lu": head["growth_lu"],
            "growth_rel_err_max": head["growth_rel_err_max"],
            "iface_pos_error_lu": head["iface_pos_error_lu"],
            "solute_drift_rel": head["solute_drift_rel"],
            "with_accumulated_bound": head["with_accumulated_bound"],
            "block_lengths": {str(k): {kk: v for kk, v in r.items()
                                       if kk not in ("training", "held_out_problem")}
                              | {"held_out_ratio": r["training"]["held_out_ratio"],
                                 "validation": r["training"]["validation"]}
                              for k, r in arms.items()},
            "roofline": {"bound": "tensor", "achieved": tflops, "peak": peak_tf,
                         "unit": "TFLOP/s", "frac": tflops / peak_tf, "peak_source": peak_kind,
                         "traffic": None, "kernel": "network forward (17 conv3x3_tc + 2 "
                         "element-wise launches), 512x512, batch 1",
                         "algorithmic_flops_per_forward": flop, "forward_ms": fwd_ms},
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": "MLUPS",
                    "h2d_bytes_per_step": int(hs.numel()) / (Ke * nb),
                    "d2h_bytes_per_step": int(ho.numel()) * 4 / (Ke * nb)},
            "gpu_launches": launches,
            "clocks": clk.summary(),
        }
        print(json.dumps(out), flush=True)
    for x in (a, net):
        x.close()
    if dist is not None:
        dist.destroy_process_group()

if __name__ == "__main__":
    main()
