"""Benchmark of the hot path: Fig. 1's time step on a virtual 2x2x2 topology
of 512x256x256 FP64 subdomains (overlap 2, periodic in x) held in one GPU,
with the halo update hidden behind the inner block (widths (16, 2, 2)).

One step = boundary slabs + halo update of T2 (high-priority stream) and the
inner block (low-priority stream), then the swap; K steps run as CUDA-graph
launches. Metric: T_eff = 3*N*s / t_step (read T and Ci, write T2, N all
points of all subdomains, s bytes per element) in GB/s, and cell updates/s.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

With torchrun (N > 1) every rank runs its own replica of the workload on its
GPU (weak scaling, no data-path collective); the timing is the maximum over
ranks. `--impl reference` times the FP64 CPU oracle on a bounded sample of the
same workload on this machine's host cores (rank 0 only).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

METRIC = "T_eff GB/s per step (3*N*s bytes / step time), stencil + halo, hidden communication"
WORKLOAD = "decomposed_2x2x2_512x256x256"


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def dist_max(x: float, ws: int, device="cuda") -> float:
    """Maximum of x over the ranks (the slowest rank's time)."""
    if ws <= 1:
        return x
    t = torch.tensor([x], dtype=torch.float64, device=device)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


class ClockSampler:
    """nvidia-smi clock/throttle sampling while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax = float(parts[2])
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


KERNEL_SOURCES = ("tma.cu", "tma_util.cuh", "cell.cuh", "igg_internal.h", "runtime.cu")


def kernel_source_sha256() -> str:
    """Hash of the sources of the stencil kernel the roofline reports and of
    the runtime that builds its tile tables and arguments."""
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        h.update(open(os.path.join(ROOT, "paper_2211_15716_gb300", "csrc", f), "rb").read())
    return h.hexdigest()


TRAFFIC_JSON = os.path.join(ROOT, "profiles", "traffic.json")


def traffic_for(key: str, path: str = TRAFFIC_JSON):
    """DRAM bytes per launch from the committed ncu summary, or None when the
    kernel sources changed since the counters were taken."""
    try:
        with open(path) as f:
            rec = json.load(f)[key]
        if kernel_source_sha256() != rec["source_sha256"]:
            return None
        return float(rec["dram_bytes_per_launch"])
    except Exception:
        return None


_UNIT = {"byte": 1.0, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9, "Tbyte": 1e12,
         "KB": 1e3, "MB": 1e6, "GB": 1e9}


def record_traffic(csv_path: str, key: str, kernel: str, scale: float, how: str,
                   path: str = TRAFFIC_JSON) -> dict:
    """Writes profiles/traffic.json[key] from an ncu raw-page CSV export
    (ncu -i <rep> --page raw --csv): the mean over the launches of `kernel`
    (a substring of the kernel name) of dram__bytes_read.sum +
    dram__bytes_write.sum, times `scale` (captured case -> bench launch),
    with the hash of the current kernel sources, so that the figure is
    dropped from the bench line as soon as those sources change."""
    import csv
    with open(csv_path, newline="") as f:
        rows = list(csv.reader(f))
    head = rows[0]
    units = rows[1]
    ik = head.index("Kernel Name")
    ir, iw = head.index("dram__bytes_read.sum"), head.index("dram__bytes_write.sum")
    tot = []
    for r in rows[2:]:
        if len(r) <= max(ik, ir, iw) or kernel not in r[ik]:
            continue
        b = float(r[ir].replace(",", "")) * _UNIT[units[ir]] + \
            float(r[iw].replace(",", "")) * _UNIT[units[iw]]
        tot.append(b)
    if not tot:
        raise SystemExit(f"no launch of {kernel} in {csv_path}")
    try:
        with open(path) as f:
            rec = json.load(f)
    except FileNotFoundError:
        rec = {}
    mean = sum(tot) / len(tot)
    rec[key] = {"source_sha256": kernel_source_sha256(),
                "dram_bytes_per_launch": int(round(mean * scale)),
                "captured_bytes_per_launch": int(round(mean)), "launches": len(tot),
                "scale": scale, "how": how}
    with open(path, "w") as f:
        json.dump(rec, f, indent=2)
        f.write("\n")
    return rec[key]


def oracle_baseline(budget_s: float = 12.0):
    """FP64 CPU oracle, one 512x256x256 subdomain of the workload, repeated
    steps for about `budget_s` seconds on all host cores."""
    import oracle
    import synth

    oracle.build()
    cores = oracle.set_threads(os.cpu_count() or 1)
    n = (512, 256, 256)
    dims, periods, o = (2, 2, 2), (1, 0, 0), (2, 2, 2)
    ng = oracle.global_size(n, dims, o, periods)
    g = oracle.global_indices(n, dims, o, periods, 0)
    T = np.ascontiguousarray(synth.gaussian_bump(*g, ng) * np.ones((n[2], n[1], n[0])))
    Ci = np.ascontiguousarray(synth.ci_uniform_c0(1, *g, ng))
    dd = [oracle.spacing(1.0, ng[d]) for d in range(3)]
    dt = oracle.cfl_dt(*dd, 1.0, Ci.max())
    T2 = T.copy()
    reps, t0 = 0, time.perf_counter()
    while True:
        oracle.step(T2, T, Ci, 1.0, dt, *dd)
        T, T2 = T2, T
        reps += 1
        el = time.perf_counter() - t0
        if el >= budget_s or reps >= 2000:
            break
    npts = n[0] * n[1] * n[2]
    inner = (n[0] - 2) * (n[1] - 2) * (n[2] - 2)
    return {"value": 3 * npts * 8 * reps / el / 1e9, "unit": "GB/s", "cores": cores, "kind": "oracle",
            "sample": f"{reps} steps of one 512x256x256 FP64 subdomain (of 8), no halo, {el:.1f} s",
            "cell_updates_per_s": inner * reps / el}


def grid_launches_per_step(grid, dtype="f64", f64_emu=True) -> int:
    """Kernel launches of one step of the default hidden form: the stencil
    launch, the emulated FP64 cell's fix-up launch (FP64 fields), and the
    one-launch halo update of 3-D grids with neighbours."""
    n = 1 + (1 if dtype == "f64" and f64_emu else 0)
    dims, periods = grid.dims, grid.periods
    if any(dims[d] > 1 or periods[d] for d in range(3)):
        n += 1
    return n


def run_launches(grid, dtype, steps) -> int:
    """Kernel launches of a run of `steps` steps of the bench grid: FP32 and
    BF16 runs of four steps or more update the halo in the last two only."""
    n = grid_launches_per_step(grid, dtype) * steps
    if dtype != "f64" and steps >= 4 and grid_launches_per_step(grid, dtype) > 1:
        n -= steps - 2
    return n


def run_reference(args, ws, rank):
    if rank != 0:
        return 0
    cb = oracle_baseline(budget_s=max(5.0, min(60.0, 2.0 * (args.steps + args.warmup))))
    line = {"impl": "reference", "metric": METRIC, "value": cb["value"], "unit": "GB/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": None, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "sample": cb["sample"]},
            "cpu_baseline": cb,
            "e2e": {"value": cb["value"], "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ---------------------------------------------------------------------------
# --forms: the reduced-precision, batched and adjoint forms, each against the
# FP64 form on the same GPU, one JSON line each (not the headline line)
# ---------------------------------------------------------------------------
def step_samples(fn, n, stream, steps_per_call):
    """n timed calls of fn (each steps_per_call steps) back to back: the
    median ms per step and the 95 % confidence interval of the median from
    the order statistics at ranks n/2 -+ 1.96 sqrt(n)/2."""
    import torch as _t
    evs = [(_t.cuda.Event(enable_timing=True), _t.cuda.Event(enable_timing=True)) for _ in range(n)]
    for a, b in evs:
        a.record(stream)
        fn()
        b.record(stream)
    _t.cuda.synchronize()
    t = [a.elapsed_time(b) / steps_per_call for a, b in evs]
    med, lo, hi = median_ci95(t)
    return {"n": n, "steps_per_sample": steps_per_call, "median_ms_per_step": round(med, 4),
            "ci95_ms_per_step": [round(lo, 4), round(hi, 4)],
            "min_ms_per_step": round(min(t), 4), "max_ms_per_step": round(max(t), 4)}


def median_ci95(samples):
    """Median of the samples and the distribution-free 95 % confidence
    interval of the median: the order statistics at ranks n/2 -+ 1.96 sqrt(n)/2
    (1-based, rounded outward, clamped to the sample)."""
    t = sorted(samples)
    n = len(t)
    half = 1.959964 * math.sqrt(n) / 2
    lo = max(0, int(math.floor(n / 2 - half)) - 1)
    hi = min(n - 1, int(math.ceil(n / 2 + half)) - 1)
    med = 0.5 * (t[(n - 1) // 2] + t[n // 2])
    return med, t[lo], t[hi]


def _timed(fn, reps):
    import torch as _t
    fn()
    _t.cuda.synchronize()
    a, b = _t.cuda.Event(enable_timing=True), _t.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(reps):
        fn()
    b.record()
    _t.cuda.synchronize()
    return a.elapsed_time(b) / reps


def form_precision(steps):
    """1024^3 grid, T0 = 1.7 + 8 sine modes, Ci ~ U[0.4, 0.67]: ms/step and
    T_eff per storage type; error against the FP64 oracle after 1000 steps at
    128^3 with the same recipe. The timed 1024^3 fields are evaluated on the
    device from the same recipe (the seeded mode numbers, one outer product
    per mode; Ci from a seeded device generator): their values may differ
    from the host generators' in the last bits, which the timing does not
    depend on; the accuracy check uses the host generators."""
    import oracle
    import synth
    import paper_2211_15716_gb300 as igg
    from paper_2211_15716_gb300 import workloads as wl

    out = {"form": "precision", "workload": "1024^3 single grid, sine modes, nt timed " + str(steps)}
    n = 1024
    w = wl.WORKLOADS["precision_1024"]
    g = igg.Grid((n, n, n))
    res = {}
    gen = torch.Generator(device="cuda").manual_seed(w.seed)
    C64 = torch.rand(g.shape, dtype=torch.float64, device="cuda", generator=gen) * 0.27 + 0.4
    dx, dy, dz, dt = wl.setup(w, g, C64)
    x = torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1)
    T64 = torch.full(g.shape, 1.7, dtype=torch.float64, device="cuda")
    for mx, my, mz in synth.sine_mode_numbers(w.seed):
        sx, sy, sz = (torch.sin(math.pi * int(m) * x) for m in (mx, my, mz))
        T64[0] += 0.1 * (sz[:, None, None] * sy[None, :, None]) * sx[None, None, :]

    def storage(x, tdt):  # FP64 -> FP32 -> BF16, each nearest-even (the inputs' definition)
        return x if tdt == torch.float64 else (x.float() if tdt == torch.float32 else x.float().to(tdt))

    for name, tdt in (("f64_emulated", torch.float64), ("f64_cell", torch.float64),
                      ("f32", torch.float32), ("bf16", torch.bfloat16)):
        T = storage(T64, tdt).clone()
        Ci = storage(C64, tdt)
        T2 = T.clone()
        g.set_option(g.OPT_F64_EMU, 0 if name == "f64_cell" else 1)
        ms = _timed(lambda: g.run(steps, T, T2, Ci, w.lam, dt, dx, dy, dz), 1) / steps
        nb = 3 * n ** 3 * T.element_size()
        res[name] = {"ms_per_step": round(ms, 4), "T_eff_GB_s": round(nb / (ms * 1e-3) / 1e9, 1),
                     "cell_updates_per_s": (n - 2) ** 3 / (ms * 1e-3)}
        del T, T2, Ci
        torch.cuda.empty_cache()
    g.set_option(g.OPT_F64_EMU, 1)
    g.finalize()
    del C64, T64
    # accuracy at 128^3, nt = 1000, against the FP64 oracle
    m, nt = 128, 1000
    wa = wl.WORKLOADS["precision_128"]
    ga = igg.Grid((m, m, m))
    T0, Ci = wl.host_fields(wa, ga, 0)
    T0, Ci = np.ascontiguousarray(T0), np.ascontiguousarray(Ci)
    dd = [oracle.spacing(1.0, m)] * 3
    dt_o = oracle.cfl_dt(*dd, 1.0, Ci.max())
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    ref = oracle.run(T0, Ci, nt, 1.0, dt_o, *dd)
    scale = np.abs(ref).max()
    errs = {}
    for name, tdt, emu in (("f64_emulated", torch.float64, 1), ("f64_cell", torch.float64, 0),
                           ("f32", torch.float32, 1), ("bf16", torch.bfloat16, 1)):
        T, T2, Cd = wl.make_fields(wa, ga, tdt)
        ga.set_option(ga.OPT_F64_EMU, emu)
        r = ga.run(nt, T, T2, Cd, 1.0, dt_o, *dd).double().cpu().numpy()[0]
        d = r - ref
        errs[name] = {"max_abs_err_rel_to_max_T": float(np.abs(d).max() / scale),
                      "rel_L2": float(np.linalg.norm(d) / np.linalg.norm(ref))}
    errs["change_of_T_over_run_rel"] = float(np.abs(ref - T0).max() / scale)
    ga.finalize()
    out.update({"results": res, "error_vs_fp64_oracle_128cube_nt1000": errs})
    return out


def form_batched(steps):
    """256 independent FP32 problems, dims uniform on {32..192}: one launch
    per step, CUDA-graph loop, autotuned kernel and tiling."""
    import oracle
    import synth
    import paper_2211_15716_gb300 as igg
    from paper_2211_15716_gb300 import workloads as wl

    sizes, lam, ci, dd, dt = wl.batch_problems()
    B = igg.Batch(sizes, torch.float32)
    B.set_coefs(lam, dt, [d[0] for d in dd], [d[1] for d in dd], [d[2] for d in dd])
    T, T2, Ci = wl.make_batch_fields(B, ci)
    best = B.autotune(T2, T, Ci, reps=3)
    T2.copy_(T)
    ms = _timed(lambda: B.run(steps, T, T2, Ci), 1) / steps
    cells = sum(a * b * c for a, b, c in sizes)
    inner = sum((a - 2) * (b - 2) * (c - 2) for a, b, c in sizes)
    # accuracy: 4 sampled problems after 200 steps against the oracle
    T, T2, Ci = wl.make_batch_fields(B, ci)
    nt = 200
    res = B.run(nt, T, T2, Ci)
    torch.cuda.synchronize()
    worst = 0.0
    for b in (0, 63, 128, 255):
        nx, ny, nz = sizes[b]
        g = [np.arange(nx), np.arange(ny), np.arange(nz)]
        T0 = np.ascontiguousarray(np.broadcast_to(synth.gaussian_bump(*g, (nx, ny, nz)), (nz, ny, nx)))
        ref = oracle.run(T0, np.full(T0.shape, float(ci[b])), nt, float(lam[b]), dt[b], *dd[b])
        gpu = B.view(res, b).double().cpu().numpy()
        worst = max(worst, float(np.abs(gpu - ref).max() / np.abs(ref).max()))
    B.destroy()
    return {"form": "batched", "workload": "256 FP32 problems, dims U{32..192}, lam U[0.5,2]",
            "ms_per_step": round(ms, 4), "T_eff_GB_s": round(3 * cells * 4 / (ms * 1e-3) / 1e9, 1),
            "cell_updates_per_s": inner / (ms * 1e-3), "cells": cells, "autotuned": best,
            "max_err_rel_vs_fp64_oracle_nt200_4problems": worst}


def form_adjoint():
    """256^3 FP64 and FP32, nt = 200, misfit gradient through the checkpointed
    adjoint (checkpoint every 16): time against the plain forward run, and a
    central finite difference of J along a random direction of Ci."""
    import synth
    import paper_2211_15716_gb300 as igg
    from paper_2211_15716_gb300 import autograd as ag
    from paper_2211_15716_gb300 import workloads as wl

    n, nt, every = 256, 200, 16
    g = igg.Grid((n, n, n))
    gi = [np.arange(n)] * 3
    out = {"form": "adjoint", "workload": "256^3, nt 200, checkpoint every 16"}
    Ci_star = synth.ci_smooth(4, *gi, (n, n, n))
    T0 = np.broadcast_to(synth.gaussian_bump(*gi, (n, n, n), sigma=0.15), (n, n, n))
    dd = [wl.spacing(1.0, n)] * 3
    dt = wl.cfl_dt(*dd, 1.0, max(Ci_star.max(), 0.53))
    noise = 1e-3 * synth.normal(4, 20, np.arange(n ** 3, dtype=np.uint64)).reshape(n, n, n)
    for name, tdt in (("f64", torch.float64), ("f32", torch.float32)):
        cs = torch.from_numpy(np.ascontiguousarray(Ci_star)).to(tdt).cuda().view(g.shape)
        t0 = torch.from_numpy(np.ascontiguousarray(T0)).to(tdt).cuda().view(g.shape)
        obs = g.run(nt, t0.clone(), t0.clone(), cs, 1.0, dt, *dd)
        obs = obs + torch.from_numpy(noise).to(tdt).cuda().view(g.shape)
        C = torch.full(g.shape, 0.53, dtype=tdt, device="cuda")
        t_fwd = _timed(lambda: g.run(nt, t0.clone(), t0.clone(), C, 1.0, dt, *dd), 2)

        def grad():
            T_nt, ck = ag.forward_checkpointed(g, nt, every, t0, C, 1.0, dt, *dd)
            lam_nt = ag.residual(T_nt, obs)
            return ag.adjoint_checkpointed(g, nt, every, ck, C, lam_nt, 1.0, dt, *dd)

        t_grad = _timed(grad, 2)
        gT, gC = grad()
        # one adjoint step on its own: lam_in, Ci, T_n read, lam_out written,
        # gCi (FP64) read and written
        Tn = g.run(nt // 2, t0.clone(), t0.clone(), C, 1.0, dt, *dd)
        lam_in = obs - Tn
        lam_out = torch.empty_like(lam_in)
        gci = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        t_adj = _timed(lambda: ag.adjoint_step(g, lam_out, lam_in, Tn, C, gci, 1.0, dt, *dd), 20)
        adj_bytes = (4 * Tn.element_size() + 16) * n ** 3

        def J(Cx):
            T_nt = g.run(nt, t0.clone(), t0.clone(), Cx, 1.0, dt, *dd)
            return 0.5 * igg.reduce(igg.RED_SUM_SQDIFF, T_nt, obs).item()

        v = torch.from_numpy(synth.normal(4, 30, np.arange(n ** 3, dtype=np.uint64)).reshape(g.shape)).cuda()
        res = {"forward_ms": round(t_fwd, 3), "gradient_ms": round(t_grad, 3),
               "gradient_over_forward": round(t_grad / t_fwd, 2),
               "adjoint_step_ms": round(t_adj, 4),
               "adjoint_step_GB_s": round(adj_bytes / (t_adj * 1e-3) / 1e9, 1),
               "adjoint_step_frac_of_hbm": round(adj_bytes / (t_adj * 1e-3) / 1e9 / peaks()[0], 3)}
        if tdt == torch.float64:
            h = 1e-7
            fd = (J(C + (h * v).to(tdt)) - J(C - (h * v).to(tdt))) / (2 * h)
            ad = float((gC * v).sum())
            res["fd_vs_adjoint_rel"] = abs(fd - ad) / abs(ad)
            g64 = gC
        else:  # FP32 fields: compare with the FP64 gradient of the same problem
            res["rel_L2_vs_fp64_gradient_Ci"] = float((gC - g64).norm() / g64.norm())
        out[name] = res
    g.finalize()
    return out


def form_acoustic(steps):
    """Staggered-grid acoustics on 2x2x2 subdomains of 256^3 cells (cell P,
    three face fields one point longer), FP64 and FP32: ms per step with the
    halo update of all four fields, and T_eff over the 12 field passes of a
    step (velocities: read P, read and write Vx, Vy, Vz; pressure: read Vx,
    Vy, Vz, read and write P)."""
    import paper_2211_15716_gb300 as igg
    n, dims = (256, 256, 256), (2, 2, 2)
    rho, K, h = 1.0, 2.0, (1 / 511, 1 / 511, 1 / 511)
    dt = 0.3 * h[0] / math.sqrt(K / rho)
    out = {"form": "acoustic", "workload": "2x2x2 x 256^3 cells, staggered P, Vx, Vy, Vz, walls"}
    with igg.Grid(n, dims=dims, overlap=(2, 2, 2)) as g:
        cells = g.nsub * n[0] * n[1] * n[2]
        for dtype, name in ((torch.float64, "f64"), (torch.float32, "f32")):
            P, Vx, Vy, Vz = g.acoustic_fields(dtype)
            P.uniform_(-0.5, 0.5)
            step = lambda: g.acoustic_step(P, Vx, Vy, Vz, rho, K, dt, *h)  # noqa: E731
            for _ in range(3):
                step()
            ms = _timed(lambda: [step() for _ in range(steps)], 1) / steps
            s = P.element_size()
            out[name] = {"ms_per_step": round(ms, 4),
                         "T_eff_GB_s": round(12 * cells * s / (ms * 1e-3) / 1e9, 1),
                         "cell_updates_per_s": cells / (ms * 1e-3)}
            del P, Vx, Vy, Vz
    return out


def form_gp(steps):
    """Gross-Pitaevskii on 2x2x2 subdomains of 256^3 points, FP64 and FP32:
    ms per step (two half steps, each followed by the halo update of its
    field) and T_eff over the 8 field passes of a step (each half: read u, v,
    V, write the updated field)."""
    import paper_2211_15716_gb300 as igg
    n, dims = (256, 256, 256), (2, 2, 2)
    h = 1.0 / 510
    g = 1.0
    dt = 0.3 / (2 * 3 / h ** 2 + 1.0 + 2 * g)
    out = {"form": "gross_pitaevskii", "workload": "2x2x2 x 256^3, psi = u + i v, harmonic potential"}
    with igg.Grid(n, dims=dims, overlap=(2, 2, 2)) as gr:
        cells = gr.nsub * gr.nloc
        for dtype, name in ((torch.float64, "f64"), (torch.float32, "f32")):
            u = torch.rand(gr.shape, dtype=dtype, device="cuda") - 0.5
            v = torch.rand(gr.shape, dtype=dtype, device="cuda") - 0.5
            P = torch.rand(gr.shape, dtype=dtype, device="cuda")
            step = lambda: gr.gp_step(u, v, P, g, dt, h, h, h)  # noqa: E731
            for _ in range(3):
                step()
            ms = _timed(lambda: [step() for _ in range(steps)], 1) / steps
            s = u.element_size()
            out[name] = {"ms_per_step": round(ms, 4),
                         "T_eff_GB_s": round(8 * cells * s / (ms * 1e-3) / 1e9, 1),
                         "cell_updates_per_s": cells / (ms * 1e-3)}
            del u, v, P
    return out


def profile_case(which):
    """Short fixed workloads for ncu captures of one kernel (not bench lines):
    'stencil': four hidden steps (stencil launch, fix-up launch, halo update)
    of the 2x2x2 x 256x128x128 FP64 workload, the same launches as the
    benchmark's steps at one eighth of the points; 'stencil_signed': the same
    on its sign-changing field; 'adjoint': 13 adjoint
    steps at 256^3 on FP64 fields (T_n the Gaussian bump, sigma 0.15), then 13
    on FP32 fields; 'gp': three Gross-Pitaevskii steps on 2x2x2 x 128^3, FP64
    then FP32; 'stencil_groups': three plain steps of the 2x2x2 x 256x128x128
    grid with the workload's spacings (two weight groups), then three with
    equal spacings (one group), on T = 2 + U[0, 5e-4] (one binade) and
    Ci = 1/U[1.5, 2.5]; 'acoustic': three acoustic steps (velocities,
    pressure, halo update of the four fields) on 2x2x2 x 256^3 cells, FP64
    then FP32. Prints each case's ms per launch."""
    import synth
    import paper_2211_15716_gb300 as igg
    from paper_2211_15716_gb300 import autograd as ag
    from paper_2211_15716_gb300 import workloads as wl

    if which in ("stencil", "stencil_signed"):
        w = wl.WORKLOADS["decomposed_2x2x2_256x128x128" + ("_signed" if which == "stencil_signed" else "")]
        g = igg.Grid(w.n, dims=w.dims, overlap=w.overlap, periods=w.periods)
        T, T2, Ci = wl.make_fields(w, g)
        dx, dy, dz, dt = wl.setup(w, g, Ci)
        g.set_option(g.OPT_PHASE_TIMES, 1)
        for _ in range(4):
            g.step_hidden(w.widths, T2, T, Ci, w.lam, dt, dx, dy, dz)
            T, T2 = T2, T
        a, b, tot, k = g.phase_times()
        print(json.dumps({"profile": which, "stencil_phase_ms": round(a / k, 4),
                          "halo_ms": round(b / k, 4), "device_status": g.device_status()}))
        g.finalize()
    elif which == "acoustic":
        n = (256, 256, 256)
        h = (1 / 511, 1 / 511, 1 / 511)
        dt = 0.3 * h[0] / math.sqrt(2.0)
        with igg.Grid(n, dims=(2, 2, 2), overlap=(2, 2, 2)) as g:
            for tdt in (torch.float64, torch.float32):
                P, Vx, Vy, Vz = g.acoustic_fields(tdt)
                P.uniform_(-0.5, 0.5)
                ms = _timed(lambda: g.acoustic_step(P, Vx, Vy, Vz, 1.0, 2.0, dt, *h), 2)
                print(json.dumps({"profile": "acoustic", "dtype": str(tdt), "ms_per_step": round(ms, 4)}))
                del P, Vx, Vy, Vz
    elif which == "stencil_groups":
        g = igg.Grid((256, 128, 128), dims=(2, 2, 2), overlap=(2, 2, 2), periods=(1, 0, 0))
        gen = torch.Generator(device="cuda").manual_seed(0)
        T = 2.0 + 0.5 * torch.rand(g.shape, dtype=torch.float64, device="cuda", generator=gen) * 1e-3
        Ci = 1.0 / (1.5 + torch.rand(g.shape, dtype=torch.float64, device="cuda", generator=gen))
        T2 = T.clone()
        ng = g.global_size()
        for name, (dx, dy, dz) in (("two groups", (1 / (ng[0] - 1), 1 / (ng[1] - 1), 1 / (ng[2] - 1))),
                                   ("one group", (1 / 255, 1 / 255, 1 / 255))):
            dt = min(dx, dy, dz) ** 2 / 0.67 / 6.1
            ms = _timed(lambda: g.step(T2, T, Ci, 1.0, dt, dx, dy, dz), 2)
            print(json.dumps({"profile": "stencil_groups", "case": name, "ms_per_step": round(ms, 4)}))
        g.finalize()
    elif which == "adjoint":
        n = 256
        g = igg.Grid((n, n, n))
        gi = [np.arange(n)] * 3
        gauss = np.ascontiguousarray(np.broadcast_to(synth.gaussian_bump(*gi, (n, n, n), sigma=0.15),
                                                     (n, n, n)))
        dd = [wl.spacing(1.0, n)] * 3
        dt = wl.cfl_dt(*dd, 1.0, 0.67)
        for tdt in (torch.float64, torch.float32):
            gen = torch.Generator(device="cuda").manual_seed(0)
            lam_in = torch.randn(g.shape, dtype=torch.float64, device="cuda", generator=gen).to(tdt)
            Tn = torch.from_numpy(gauss).to(tdt).cuda().view(g.shape).contiguous()
            C = torch.full(g.shape, 0.53, dtype=tdt, device="cuda")
            out = torch.empty_like(lam_in)
            gci = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
            ms = _timed(lambda: ag.adjoint_step(g, out, lam_in, Tn, C, gci, 1.0, dt, *dd), 12)
            print(json.dumps({"profile": "adjoint", "dtype": str(tdt), "ms_per_launch": round(ms, 4),
                              "device_status": g.device_status()}))
        g.finalize()
    elif which == "gp":
        n = 128
        h = 1.0 / (2 * n - 2)
        gnl = 1.0
        dt = 0.3 / (2 * 3 / h ** 2 + 1.0 + 2 * gnl)
        with igg.Grid((n, n, n), dims=(2, 2, 2), overlap=(2, 2, 2)) as gr:
            for tdt in (torch.float64, torch.float32):
                gen = torch.Generator(device="cuda").manual_seed(0)
                u = torch.rand(gr.shape, dtype=tdt, device="cuda", generator=gen) - 0.5
                v = torch.rand(gr.shape, dtype=tdt, device="cuda", generator=gen) - 0.5
                P = torch.rand(gr.shape, dtype=tdt, device="cuda", generator=gen)
                ms = _timed(lambda: gr.gp_step(u, v, P, gnl, dt, h, h, h), 2)
                print(json.dumps({"profile": "gp", "dtype": str(tdt), "ms_per_step": round(ms, 4),
                                  "device_status": gr.device_status()}))
    return 0


def run_forms(args):
    import paper_2211_15716_gb300  # noqa: F401
    from paper_2211_15716_gb300 import build as igg_build
    igg_build.build()
    for fn in (lambda: form_precision(max(20, args.steps // 5)), lambda: form_batched(max(20, args.steps)),
               form_adjoint, lambda: form_acoustic(max(20, args.steps // 5)),
               lambda: form_gp(max(20, args.steps // 5))):
        print(json.dumps(fn()), flush=True)
        torch.cuda.empty_cache()
    return 0


E2E_NT = 100       # steps of the end-to-end job (Fig. 1's nt)
SUSTAINED_S = 0.5  # least duration of the sustained timed block
PHASE_STEPS = 20   # eagerly queued steps timed per phase for the roofline


def timed_steps(grid, w, fields, nt, stream, widths="default"):
    """nt steps of the graph-captured loop on `stream`, CUDA-event timed:
    (ms, fields with the newest state first)."""
    T, T2, Ci, dt, dx, dy, dz = fields
    wd = w.widths if widths == "default" else widths
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    cur = grid.run(nt, T, T2, Ci, w.lam, dt, dx, dy, dz, widths=wd)
    e1.record(stream)
    torch.cuda.synchronize()
    if cur is T2:
        T, T2 = T2, T
    return e0.elapsed_time(e1), (T, T2, Ci, dt, dx, dy, dz)


def phase_ms(grid, w, fields, steps, hidden=True):
    """Per-step device time of the stencil phase (the stencil launches with
    their fix-up launches, until both tile sets end) and of the rest of the
    step (the halo update's tail), from the library's phase events around
    `steps` eagerly queued steps: the same launches, tile tables and
    arguments as the steps inside the timed graphs."""
    T, T2, Ci, dt, dx, dy, dz = fields
    grid.set_option(grid.OPT_PHASE_TIMES, 1)
    for _ in range(steps):
        if hidden:
            grid.step_hidden(w.widths, T2, T, Ci, w.lam, dt, dx, dy, dz)
        else:
            grid.step(T2, T, Ci, w.lam, dt, dx, dy, dz)
        T, T2 = T2, T
    a, b, tot, n = grid.phase_times()
    grid.set_option(grid.OPT_PHASE_TIMES, 0)
    return a / n, b / n, (T, T2, Ci, dt, dx, dy, dz)


def worst_case(args, grid, w_name, Ci, dt, dd, stream):
    """The hidden step on the sign-changing T0 (sine modes about 0), same grid,
    Ci and dt: ms per step and the share of points the emulated FP64 cell
    left to its fix-up launch."""
    from paper_2211_15716_gb300 import workloads as wl
    w = wl.WORKLOADS[w_name]
    T, T2, _ = wl.make_fields(w, grid, torch.float64)
    f = (T, T2, Ci, dt, *dd)
    _, f = timed_steps(grid, w, f, 4, stream)
    grid.fixup_stats(clear=True)
    steps = max(10, args.steps)
    ms, f = timed_steps(grid, w, f, steps, stream)
    segs, pts = grid.fixup_stats(clear=True)
    inner = grid.nsub * (w.n[0] - 2) * (w.n[1] - 2) * (w.n[2] - 2)
    bytes_step = 3 * grid.nsub * grid.nloc * 8
    a, b, f = phase_ms(grid, w, f, 6)
    del f, T, T2
    torch.cuda.empty_cache()
    return {"workload": w_name, "ms_per_step": round(ms / steps, 4),
            "GB_s": round(bytes_step / (ms / steps * 1e-3) / 1e9, 1),
            "fixup_point_share": round(pts / (steps * inner), 5),
            "fixup_segments_per_step": round(segs / steps, 1),
            "stencil_phase_ms": round(a, 4), "halo_ms": round(b, 4),
            "note": "T0 = 8 sine modes of amplitude 0.1 about 0; parity at 1e-12 in the GPU tests"}


def _storage(x, tdt):
    """FP64 -> FP32 -> BF16 storage, each rounding to nearest even (the
    inputs' definition, as synth's converters apply it)."""
    return x.float() if tdt == torch.float32 else x.float().to(tdt)


def cfg1_other_dtype(args, grid, w, tdt, dd_dt, ref64, T0_64, Ci64, stream):
    """The cfg1 hidden step with FP32 or BF16 fields (the FP64 inputs T0_64,
    Ci64 rounded to the storage type on the device): ms per step for the
    default form, the split and the halo update beside the inner tiles, and
    the error after E2E_NT steps against the FP64 GPU form (max |dT| /
    max |T|)."""
    dx, dy, dz, dt = dd_dt

    def fresh():
        T = _storage(T0_64, tdt)
        return T, T.clone(), _storage(Ci64, tdt)

    T, T2, Ci = fresh()
    f = (T, T2, Ci, dt, dx, dy, dz)
    _, f = timed_steps(grid, w, f, 4, stream)
    steps = max(10, args.steps)
    ms, f = timed_steps(grid, w, f, steps, stream)
    a, b, f = phase_ms(grid, w, f, 6)
    grid.set_option(grid.OPT_FUSED_HALO, 0)
    _, f = timed_steps(grid, w, f, 2, stream)  # tiles and graph made untimed
    ms_split, f = timed_steps(grid, w, f, steps, stream)
    grid.set_option(grid.OPT_FUSED_HALO, 1)
    grid.set_option(grid.OPT_HIDE_HALO, 1)
    _, f = timed_steps(grid, w, f, 2, stream)  # tiles and graph made untimed
    ms_hide, f = timed_steps(grid, w, f, steps, stream)
    grid.set_option(grid.OPT_HIDE_HALO, 0)
    s = T.element_size()
    bytes_step = 3 * grid.nsub * grid.nloc * s
    T, T2, Ci = fresh()
    cur = grid.run(E2E_NT, T, T2, Ci, w.lam, dt, dx, dy, dz, widths=w.widths)
    err = float((cur.double() - ref64).abs().max() / ref64.abs().max())
    del T, T2, Ci, cur, f
    torch.cuda.empty_cache()
    ms_s = ms / steps
    return {"ms_per_step": round(ms_s, 4), "GB_s": round(bytes_step / (ms_s * 1e-3) / 1e9, 1),
            "frac_of_hbm": round(bytes_step / (ms_s * 1e-3) / 1e9 / peaks()[0], 3),
            "stencil_phase_ms": round(a, 4), "halo_ms": round(b, 4),
            "split_ms_per_step": round(ms_split / steps, 4),
            "halo_beside_inner_tiles_ms_per_step": round(ms_hide / steps, 4),
            f"max_err_rel_vs_fp64_gpu_nt{E2E_NT}": err}


def compact_forms(args, budget_s):
    """The reshaped forms, each against the FP64 form on the same GPU at a
    stated accuracy, within about budget_s seconds (later forms are skipped
    once the budget is spent, and say so)."""
    out, t0 = {}, time.perf_counter()
    hbm = peaks()[0]
    jobs = (("precision_1024", lambda: form_precision(20)),
            ("batched_256", lambda: form_batched(max(20, args.steps))),
            ("adjoint_256", form_adjoint),
            ("acoustic_2x2x2x256", lambda: form_acoustic(20)),
            ("gross_pitaevskii_2x2x2x256", lambda: form_gp(20)))
    for name, fn in jobs:
        if time.perf_counter() - t0 > budget_s:
            out[name] = {"skipped": f"time budget of {budget_s:.0f} s spent"}
            continue
        t1 = time.perf_counter()
        r = fn()
        torch.cuda.empty_cache()
        r["seconds"] = round(time.perf_counter() - t1, 1)
        out[name] = _with_fracs(r, hbm)
    return out


def _with_fracs(r, hbm):
    """Adds frac_of_hbm beside every T_eff_GB_s of a form's result."""
    if isinstance(r, dict):
        for k in list(r):
            r[k] = _with_fracs(r[k], hbm)
        if "T_eff_GB_s" in r:
            r["frac_of_hbm"] = round(r["T_eff_GB_s"] / hbm, 3)
    return r


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-forms", action="store_true",
                    help="leave the reshaped forms out of the JSON line")
    ap.add_argument("--forms-budget", type=float, default=60.0,
                    help="seconds allowed for the reshaped forms")
    ap.add_argument("--workload", default=WORKLOAD,
                    help="decomposed_2x2x2_512x256x256 (default) or a smaller case for profiling")
    ap.add_argument("--dtype", default="f64", choices=["f64", "f32", "bf16"])
    ap.add_argument("--forms", action="store_true",
                    help="only measure the reshaped forms (one JSON line each)")
    ap.add_argument("--profile",
                    choices=["stencil", "stencil_signed", "stencil_groups", "adjoint", "gp", "acoustic"],
                    help="run a short fixed workload of one kernel for an ncu capture")
    ap.add_argument("--record-traffic", metavar="CSV",
                    help="write profiles/traffic.json from an ncu raw CSV export (no GPU)")
    ap.add_argument("--traffic-key", default=f"hidden step stencil f64 {WORKLOAD}")
    ap.add_argument("--traffic-kernel", default="k_stencil_tma")
    ap.add_argument("--traffic-scale", type=float, default=8.0)
    ap.add_argument("--traffic-how", default="")
    args = ap.parse_args()
    if args.record_traffic:
        print(json.dumps(record_traffic(args.record_traffic, args.traffic_key, args.traffic_kernel,
                                        args.traffic_scale, args.traffic_how)))
        return 0
    ws, rank, local = dist_env()
    if args.impl == "reference":
        return run_reference(args, ws, rank)
    if args.forms:
        return run_forms(args)
    if args.profile:
        import paper_2211_15716_gb300  # noqa: F401
        from paper_2211_15716_gb300 import build as igg_build
        igg_build.build()
        return profile_case(args.profile)
    if args.warmup < 3:
        args.warmup = 3

    import paper_2211_15716_gb300 as igg
    from paper_2211_15716_gb300 import build as igg_build
    from paper_2211_15716_gb300 import workloads as wl

    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    igg_build.build()
    headline = args.workload == WORKLOAD and args.dtype == "f64"

    w = wl.WORKLOADS[args.workload]
    tdtype = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[args.dtype]
    grid = igg.Grid(w.n, dims=w.dims, overlap=w.overlap, periods=w.periods)
    T, T2, Ci = wl.make_fields(w, grid, tdtype)
    if tdtype == torch.float64:
        dx, dy, dz, dt = wl.setup(w, grid, Ci)
    else:  # dt from the FP64 inputs, as for the FP64 form
        _, _, Ci64 = wl.make_fields(w, grid, torch.float64)
        dx, dy, dz, dt = wl.setup(w, grid, Ci64)
        del Ci64, _
    N = grid.nsub * grid.nloc
    inner = grid.nsub * (w.n[0] - 2) * (w.n[1] - 2) * (w.n[2] - 2)
    s = T.element_size()
    bytes_step = 3 * N * s
    stream = torch.cuda.current_stream()
    fields = (T, T2, Ci, dt, dx, dy, dz)

    # warm-up (also captures the two-step CUDA graph)
    _, fields = timed_steps(grid, w, fields, args.warmup, stream)

    def barrier():
        if ws > 1:
            torch.distributed.barrier()

    # ---- timed region: exactly K hidden steps ----------------------------
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    barrier()
    torch.cuda.synchronize()
    ms, fields = timed_steps(grid, w, fields, args.steps, stream)
    barrier()
    ms = dist_max(ms, ws)
    ms_step = ms / args.steps

    # ---- sustained block: the same loop for at least SUSTAINED_S seconds --
    sus_steps = max(args.steps, 2 * int(math.ceil(SUSTAINED_S / (ms_step * 1e-3) / 2)))
    barrier()
    ms_sus, fields = timed_steps(grid, w, fields, sus_steps, stream)
    barrier()
    ms_sus = dist_max(ms_sus, ws)

    # ---- dominant launch: the stencil phase of the same hidden steps ------
    k_ms, halo_ms, fields = phase_ms(grid, w, fields, PHASE_STEPS)
    clocks = sampler.stop()
    plain_k_ms, _, fields = phase_ms(grid, w, fields, PHASE_STEPS, hidden=False)

    # ---- per-sample step times: median and a 95 % confidence interval ----
    T, T2, Ci = fields[:3]
    samples = step_samples(lambda: grid.run(2, T, T2, Ci, w.lam, dt, dx, dy, dz, widths=w.widths),
                           40, stream, 2)

    # ---- variants (outside the timed region) ------------------------------
    variants = {}
    vsteps = max(10, args.steps // 2)
    _, fields = timed_steps(grid, w, fields, 2, stream, widths=None)  # graph made untimed
    t_plain, fields = timed_steps(grid, w, fields, vsteps, stream, widths=None)
    t_plain /= vsteps
    variants["plain_step_no_hiding"] = {
        "ms_per_step": round(t_plain, 4), "GB_s": round(bytes_step / (t_plain * 1e-3) / 1e9, 1),
        "note": "igg_run without widths: the same launches as the default hidden form"}
    grid.set_option(grid.OPT_HIDE_HALO, 1)
    _, fields = timed_steps(grid, w, fields, 2, stream)  # tiles and graph made untimed
    t_hid, fields = timed_steps(grid, w, fields, vsteps, stream)
    hid_k_ms, hid_halo_ms, fields = phase_ms(grid, w, fields, PHASE_STEPS)
    grid.set_option(grid.OPT_HIDE_HALO, 0)
    t_hid /= vsteps
    variants["hidden_step_halo_beside_inner_tiles"] = {
        "ms_per_step": round(t_hid, 4), "GB_s": round(bytes_step / (t_hid * 1e-3) / 1e9, 1),
        "stencil_phase_ms": round(hid_k_ms, 4), "halo_tail_ms": round(hid_halo_ms, 4),
        "note": "IGG_OPT_HIDE_HALO = 1: face tiles, then the halo update on a high-priority "
                "stream beside the inner tiles on a low-priority one"}
    grid.set_option(grid.OPT_FUSED_HALO, 0)
    _, fields = timed_steps(grid, w, fields, 2, stream)
    t_split, fields = timed_steps(grid, w, fields, vsteps, stream)
    grid.set_option(grid.OPT_FUSED_HALO, 1)
    t_split /= vsteps
    variants["hidden_step_split"] = {"ms_per_step": round(t_split, 4),
                                     "GB_s": round(bytes_step / (t_split * 1e-3) / 1e9, 1),
                                     "note": "boundary/inner split on two streams"}
    variants["plain_step_kernel"] = {
        "stencil_phase_ms": round(plain_k_ms, 4),
        "GB_s": round(bytes_step / (plain_k_ms * 1e-3) / 1e9, 1),
        "note": "igg_step (no halo): the stencil launch without the halo-carrying row ends"}
    if tdtype == torch.float64:
        grid.set_option(grid.OPT_F64_EMU, 0)
        _, fields = timed_steps(grid, w, fields, 2, stream)
        t_nat, fields = timed_steps(grid, w, fields, vsteps, stream)
        grid.set_option(grid.OPT_F64_EMU, 1)
        t_nat /= vsteps
        variants["hidden_step_fp64_cell"] = {"ms_per_step": round(t_nat, 4),
                                             "GB_s": round(bytes_step / (t_nat * 1e-3) / 1e9, 1)}
    grid.fixup_stats(clear=True)
    _, fields = timed_steps(grid, w, fields, 2, stream)
    segs, pts = grid.fixup_stats(clear=True)
    status = grid.device_status()

    # ---- end to end through the library: igg_run_host, fixed nt -----------
    T, T2, Ci = fields[:3]
    T0, _, C0 = wl.make_fields(w, grid, tdtype)
    Th = torch.empty(T.shape, dtype=T.dtype, pin_memory=True)
    Ch = torch.empty(Ci.shape, dtype=Ci.dtype, pin_memory=True)
    Th.copy_(T0)
    Ch.copy_(C0)
    del C0, _
    # one untimed call first (the pinned buffers' first transfers)
    grid.run_host(2, Th, Ch, T, T2, Ci, w.lam, dt, dx, dy, dz, widths=w.widths)
    torch.cuda.synchronize()
    Th.copy_(T0)
    torch.cuda.synchronize()
    barrier()
    x0, x1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    h0 = time.perf_counter()
    x0.record(stream)
    grid.run_host(E2E_NT, Th, Ch, T, T2, Ci, w.lam, dt, dx, dy, dz, widths=w.widths)
    x1.record(stream)
    torch.cuda.synchronize()
    wall = time.perf_counter() - h0
    barrier()
    e2e_ms = dist_max(x0.elapsed_time(x1), ws)
    ref_nt = T2 if E2E_NT % 2 else T  # the newest state on the device
    assert torch.equal(Th.view(-1)[:64].to(ref_nt.device), ref_nt.view(-1)[:64])
    want_forms = headline and rank == 0 and not args.no_forms
    ref64 = ref_nt.double().clone() if want_forms else None
    T0_64 = T0 if want_forms else None
    del T0

    hbm, hbm_kind = peaks()
    launches_per_step = grid_launches_per_step(grid, args.dtype, True)
    value = ws * bytes_step / (ms_step * 1e-3) / 1e9
    achieved = bytes_step / (k_ms * 1e-3) / 1e9
    traffic = traffic_for(f"hidden step stencil {args.dtype} {args.workload}")
    line = {
        "metric": METRIC, "value": round(value, 2), "unit": "GB/s", "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_step, 4),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": args.dtype,
        "data": "synthetic (seeded Gaussian bump T0, Ci = 1/U[1.5,2.5] on global indices)",
        "config": {"workload": args.workload, "subdomains": "x".join(map(str, w.dims)),
                   "local": "x".join(map(str, w.n)), "overlap": 2, "periods": "x",
                   "widths": list(w.widths), "nt_timed": args.steps,
                   "cells": N, "inner_cells": inner, "bytes_per_step": bytes_step,
                   "l2": f"inputs larger than L2 ({bytes_step / 1e9:.2f} GB moved per step vs 129 MB L2)",
                   "graph": "two steps per CUDA graph launch",
                   "hiding": "all subdomains in one device's memory: each hidden step is the full "
                             "step launch followed by the one-launch halo update of T2; the halo "
                             "update beside the inner tiles and the paper's boundary/inner split "
                             "are variants (both slower)"},
        "cell_updates_per_s": ws * inner / (ms_step * 1e-3),
        "frac_of_8TBs": round(value / ws / 8000.0, 4),
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": hbm, "unit": "GB/s",
                     "frac": round(achieved / hbm, 4), "traffic": traffic,
                     "kernel": (f"k_stencil_tma<{args.dtype}> + k_fixup_f64 (the stencil phase of "
                                "the timed hidden step: same launches, tiles and row-end stores), "
                                "CUDA events around each step's stencil phase, "
                                f"{PHASE_STEPS} steps"),
                     "algorithmic_bytes_per_launch": bytes_step,
                     "peak_kind": hbm_kind, "kernel_ms": round(k_ms, 4),
                     "halo_update_ms": round(halo_ms, 4)},
        "sustained": {"steps": sus_steps, "seconds": round(ms_sus * 1e-3, 3),
                      "ms_per_step": round(ms_sus / sus_steps, 4),
                      "value": round(ws * bytes_step / (ms_sus / sus_steps * 1e-3) / 1e9, 2)},
        "e2e": {"value": round(ws * bytes_step * E2E_NT / (e2e_ms * 1e-3) / 1e9, 2), "unit": "GB/s",
                "nt": E2E_NT, "ms": round(e2e_ms, 3), "wall_s": round(wall, 4),
                "h2d_bytes_per_step": int(2 * N * s // E2E_NT),
                "d2h_bytes_per_step": int(N * s // E2E_NT),
                "note": (f"igg_run_host: H2D of T0 and Ci from pinned memory, T2 = copy(T) on the "
                         f"device, {E2E_NT} steps, D2H of the result, one C-ABI call")},
        "gpu_launches": run_launches(grid, args.dtype, args.steps),
        "gpu_launches_per_step": launches_per_step,
        "clocks": clocks,
        "variants": variants,
        "step_samples": samples,
        "device_status": status,
    }
    if tdtype == torch.float64:
        line["f64_cell"] = ("emulated: exact integer second differences from the bit patterns, "
                            "float-pair weighted sums, one FP64 FMA and an integer ulp correction "
                            "per point; other stencils (sign changes, powers of two crossed) in "
                            "the fix-up launch")
        line["fixup_point_share"] = round(pts / (2 * inner), 6)
    if headline:
        line["variants"]["worst_case_sign_changing_field"] = worst_case(
            args, grid, WORKLOAD + "_signed", fields[2], dt, (dx, dy, dz), stream)
    if rank == 0 and ws == 1 and not args.no_cpu_baseline and args.workload == WORKLOAD:
        line["cpu_baseline"] = oracle_baseline()
    if headline and rank == 0 and not args.no_forms:
        forms = {}
        t_f = time.perf_counter()
        for name, tdt in (("cfg1_f32", torch.float32), ("cfg1_bf16", torch.bfloat16)):
            forms[name] = cfg1_other_dtype(args, grid, w, tdt, (dx, dy, dz, dt), ref64, T0_64,
                                           fields[2], stream)
        del ref64, T0_64
        grid.finalize()
        grid = None
        del fields, T, T2, Ci
        torch.cuda.empty_cache()
        left = args.forms_budget - (time.perf_counter() - t_f)
        forms.update(compact_forms(args, max(0.0, left)))
        forms["seconds"] = round(time.perf_counter() - t_f, 1)
        line["forms"] = forms
    if rank == 0:
        print(json.dumps(line), flush=True)
    if grid is not None:
        grid.finalize()
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
