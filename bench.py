#!/usr/bin/env python3
"""Benchmark of the fused hot path on one GB300 (or N GPUs, weak scaling).

Default workload: Black-Scholes call+put pricing of 2^26 FP32 options issued
as the 23-task array program, fused by the runtime into one sm_103a kernel.
One step = issue the task window through the API + flush + the fused kernel,
inputs resident in HBM (1.34 GB per step, larger than the 129 MB L2, so no
flush of L2 is needed between steps).  Also measured in the same run: the
unfused per-task path (23 kernels, every temporary in HBM), the fused
one-kernel-per-fused-task path, the end-to-end path with host buffers (H2D of
S, K, T and D2H of call, put every step), and the CPU oracle on a bounded
sample.  Kernel durations come from CUDA events the runtime records
immediately around each launch on the launching stream.

  python bench.py [--steps K] [--warmup W] [--workload bs|cg|jacobi|batched|serve] [--fp32]
  python bench.py --impl reference     # the CPU oracle as the reference arm
Prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

# the CPU oracle is timed on one core: keep BLAS single-threaded
for _v in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

import numpy as np  # noqa: E402

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2406_18109_gb300 import configs  # noqa: E402
from synth import inputs  # noqa: E402

METRIC = {"bs": ("Black-Scholes options/s (fused window, 2^26 FP32)", "options/s", "f32"),
          "cg": ("CG iterations/s (fused windows, 256^2 Poisson FP64)", "iterations/s", "f64"),
          "jacobi": ("Jacobi sweeps/s (fused windows, 8192^2 FP32)", "sweeps/s", "f32"),
          "batched": ("Batched CG aggregate iterations/s (256 uneven solves, one launch per iteration)",
                      "iterations/s", "f64"),
          "serve": ("Serving sustained requests/s with p50/p99 latency (CG/BiCGSTAB on 3-D Poisson 64^3..256^3 "
                    "tol 1e-8, Black-Scholes 2^16..2^24; Poisson arrivals, mean gap 2 ms)", "requests/s", "f64+f32")}
WORKLOAD = {"bs": "black-scholes-2^26-fp32", "cg": "cg-poisson2d-256x256-fp64-50it",
            "jacobi": "jacobi-fig1-stencil-8192x8192-fp32-200sweeps",
            "batched": "batched-cg-256-uneven-100it",
            "serve": "serving-cg-bicgstab-bs-poisson-arrivals-2ms-120GB"}


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return {"hbm_gbs": d.get("hbm_gbs", 6800.0), "source": "measured"}
    return {"hbm_gbs": 6800.0, "source": "fallback"}


def host_link_peak(torch, mib: int = 256, reps: int = 3) -> dict:
    """Measured host<->device copy bandwidth (GB/s): pinned-host copies each
    way alone, and both ways at once on two streams (the ceiling of an end to
    end step that both uploads and downloads).  Best of `reps`."""
    n = mib << 20
    h_in = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    h_out = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    d_in = torch.empty(n, dtype=torch.uint8, device="cuda")
    d_out = torch.zeros(n, dtype=torch.uint8, device="cuda")
    s0, s1 = torch.cuda.Stream(), torch.cuda.Stream()
    best = {"h2d": 0.0, "d2h": 0.0, "both": 0.0}

    def timed(fn):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        fn()
        torch.cuda.synchronize()
        return time.perf_counter() - t0

    def both():
        with torch.cuda.stream(s0):
            d_in.copy_(h_in, non_blocking=True)
        with torch.cuda.stream(s1):
            h_out.copy_(d_out, non_blocking=True)
    for _ in range(reps + 1):
        best["h2d"] = max(best["h2d"], n / timed(lambda: d_in.copy_(h_in, non_blocking=True)) / 1e9)
        best["d2h"] = max(best["d2h"], n / timed(lambda: h_out.copy_(d_out, non_blocking=True)) / 1e9)
        best["both"] = max(best["both"], 2 * n / timed(both) / 1e9)
    del h_in, h_out, d_in, d_out
    return best


class Clocks:
    """Samples nvidia-smi during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.t.join(timeout=2)
        sm, mx, pw, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 8:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
                pw.append(float(f[3]))
            except ValueError:
                continue
            for nm, v in zip(names, f[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "power_w_max": max(pw) if pw else None, "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------ oracle
def _oracle_worker(job):
    """One host core running the oracle on its own copy of the workload's
    sample for budget_s; returns (units done, seconds)."""
    workload, seed, budget_s = job
    from oracle import programs
    done, t0 = 0, time.perf_counter()
    if workload == "bs":
        cfg = configs.BLACK_SCHOLES
        m = 1 << 20
        S, K, T = inputs.bs_inputs(m, seed=seed)
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < budget_s:
            programs.black_scholes(S, K, T, cfg["r"], cfg["sigma"], np.float32)
            done += m
    elif workload == "cg":
        cfg = configs.CG
        rp, col, val, xs = inputs.cg_inputs(m=cfg["m"], seed=seed)
        b = programs.spmv(rp, col, val, xs)
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < budget_s:
            programs.cg(rp, col, val, b, 10)
            done += 10
    else:
        cfg = configs.JACOBI
        g = inputs.jacobi_grid(2046, seed=seed)
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < budget_s:
            programs.jacobi(g, 2, np.float32)
            done += 2
    return done, time.perf_counter() - t0


ALL_CORES_SAMPLE = {
    "bs": "independent 2^20-option batches, one process per host core",
    "cg": "independent 256^2 Poisson CG solves (10 iterations at a time), one process per host core",
    "jacobi": "independent 2048^2 grids, one process per host core, sweeps scaled by area to 8192^2",
}


def oracle_rate_all_cores(workload: str = "bs", budget_s: float = 8.0):
    """The oracle on every host core at once: independent problems in spawned
    processes, BLAS single-threaded in each (the workload's weak-scaling rate
    on the host)."""
    import multiprocessing as mp
    n = os.cpu_count() or 1
    with mp.get_context("spawn").Pool(n) as pool:
        res = pool.map(_oracle_worker, [(workload, 1000 + i, budget_s) for i in range(n)])
    rate = sum(d for d, _ in res) / max(t for _, t in res)
    if workload == "jacobi":
        rate *= (2046 * 2046) / (configs.JACOBI["N"] * configs.JACOBI["N"])
    return rate, n


def oracle_rate(workload: str, budget_s: float = 10.0):
    """CPU oracle throughput on a bounded sample (the reference / cpu_baseline)."""
    from oracle import programs
    t_end = time.perf_counter() + budget_s
    if workload == "bs":
        cfg = configs.BLACK_SCHOLES
        m = 1 << 20
        S, K, T = inputs.bs_inputs(m, seed=cfg["seed"])
        done, t0 = 0, time.perf_counter()
        while True:
            programs.black_scholes(S, K, T, cfg["r"], cfg["sigma"], np.float32)
            done += m
            if time.perf_counter() > t_end:
                break
        dt = time.perf_counter() - t0
        return done / dt, "options/s", f"{done} options in batches of 2^20 drawn like the 2^26 workload (seed 1)"
    if workload == "cg":
        cfg = configs.CG
        rp, col, val, xs = inputs.cg_inputs(m=cfg["m"], seed=cfg["seed"])
        b = programs.spmv(rp, col, val, xs)
        done, t0 = 0, time.perf_counter()
        while True:
            programs.cg(rp, col, val, b, 10)
            done += 10
            if time.perf_counter() > t_end:
                break
        dt = time.perf_counter() - t0
        return done / dt, "iterations/s", f"{done} CG iterations on the 256^2 Poisson system"
    if workload == "batched":
        cfg = configs.BATCHED_CG
        dtp = np.float64 if cfg["dtype"] == "f64" else np.float32
        specs = inputs.batched_cg_problems(cfg["count"], cfg["seed"])
        rng = np.random.default_rng(0)
        sample = sorted(rng.choice(len(specs), 12, replace=False).tolist())
        t_sample, done = 0.0, 0
        for i in sample:
            rp, col, val, xs = inputs.batched_cg_matrix(specs[i])
            b = programs.spmv(rp, col, val, xs, dtp)
            t0 = time.perf_counter()
            programs.cg(rp, col, val, b, 5, dt=dtp)
            t_sample += (time.perf_counter() - t0) / 5
            done += 5
        # one iteration of every solve, estimated from the sampled solves
        per_batch = t_sample / len(sample) * len(specs)
        return len(specs) / per_batch, "iterations/s", (f"{done} CG iterations on 12 sampled problems of the "
                                                        f"batch; one iteration of all {len(specs)} solves "
                                                        f"estimated from their mean")
    if workload == "serve":
        cfg = configs.SERVING
        m0 = inputs.SERVE_LADDER[0]
        rp, col, val = inputs.poisson3d_csr(m0)
        b = programs.spmv(rp, col, val, inputs.uniform(1, -1.0, 1.0, m0 ** 3))
        hist = []
        n_run = 400
        t0 = time.perf_counter()
        programs.cg(rp, col, val, b, n_run, history=hist)
        t_it = (time.perf_counter() - t0) / n_run
        bn = np.linalg.norm(b)
        n_cg = next((k + 1 for k, x in enumerate(hist)
                     if np.linalg.norm(b - programs.spmv(rp, col, val, x)) <= cfg["tol"] * bn), n_run)
        t_cg = t_it * n_cg
        t0 = time.perf_counter()
        _, n_bi, _ = programs.bicgstab(rp, col, val, b, cfg["tol"], 2000)
        t_bi = time.perf_counter() - t0
        nb = 1 << 18
        S, K, T = inputs.bs_inputs(nb, seed=1)
        t0 = time.perf_counter()
        programs.black_scholes(S, K, T, 0.02, 0.3, np.float32)
        t_opt = (time.perf_counter() - t0) / nb
        reqs = inputs.serving_requests(cfg["count"], seed=cfg["seed"], mean_gap_s=cfg["mean_gap_ms"] * 1e-3)
        tot = 0.0
        for r in reqs:
            if r["kind"] == "bs":
                tot += t_opt * r["size"]
            else:
                # unknowns grow as m^3 and Krylov iterations on Poisson as m
                tot += (t_cg if r["kind"] == "cg" else t_bi) * (r["size"] / m0) ** 4
        return len(reqs) / tot, "requests/s", (
            f"CG ({n_cg} iterations) and BiCGSTAB ({n_bi}) solved to tol on the {m0}^3 operator, 2^18 options; "
            f"each of the {len(reqs)} requests of the stream costed from these (solves scaled by (m/{m0})^4: "
            f"m^3 unknowns x iterations growing as m), run back to back on one core")
    cfg = configs.JACOBI
    g = inputs.jacobi_grid(2046, seed=cfg["seed"])
    done, t0 = 0, time.perf_counter()
    while True:
        programs.jacobi(g, 2, np.float32)
        done += 2
        if time.perf_counter() > t_end:
            break
    dt = time.perf_counter() - t0
    scale = (2046 * 2046) / (cfg["N"] * cfg["N"])
    return done / dt * scale, "sweeps/s", f"{done} sweeps of a 2048^2 grid, scaled by area to 8192^2"


# ---------------------------------------------------------------- GPU arms
def kernel_delta(before: dict, after: dict) -> dict:
    out = {}
    for k, v in after.items():
        b = before.get(k, {"ms": 0.0, "launches": 0})
        n = v["launches"] - b["launches"]
        if n > 0:
            out[k] = {"ms": v["ms"] - b["ms"], "launches": n}
    return out


def kernel_name_of(rt):
    """Name of the generated kernel of the context's most recent launch (a
    hash of its body, so it changes whenever the generated code does)."""
    import re
    m = re.search(r"\b(dfs_[kb][0-9a-f]{16})\b", rt.kernel_source())
    return m.group(1) if m else None


class Arm:
    """One timed configuration of a workload: build state, warm up, time K steps."""

    def __init__(self, workload, rt_kwargs, torch, stream, e2e=False, graph=False, per_solve=False,
                 autotune=False):
        from paper_2406_18109_gb300 import arrays as A
        from paper_2406_18109_gb300 import workloads as W
        self.A, self.W, self.torch, self.stream, self.e2e = A, W, torch, stream, e2e
        self.per_solve, self.graph_mode, self.autotune, self.rt_kwargs = per_solve, graph, autotune, rt_kwargs
        self.tuned = None
        self.rt = A.Runtime(device=torch.cuda.current_device(), stream=stream.cuda_stream,
                            time_launches=True, **rt_kwargs)
        self.h2d = self.d2h = 0
        self.kernel_name = None
        {"bs": self._setup_bs, "cg": self._setup_cg, "batched": self._setup_batched,
         "jacobi": self._setup_jacobi}[workload]()
        self.rt.sync()
        self.keep = None

    # ------------------------------------------------------------- helpers
    def _pin(self, a):
        return self.torch.from_numpy(a).pin_memory().numpy()

    def _tune(self, step, space, key, reps, what):
        """Autotunes the context for `step`, caching the choice per GPU and key."""
        import tempfile
        from paper_2406_18109_gb300 import autotune as AT
        best, trials = AT.tune(self.rt, step, space=space, warmup=1, reps=reps, key=key,
                               cache_path=os.path.join(tempfile.gettempdir(), "dfs_autotune.json"),
                               gpu=self.torch.cuda.get_device_name())
        self.tuned = {"config": best, "trials": [{"config": c, what: m} for c, m in trials]}

    # ------------------------------------------------------------ workloads
    def _setup_bs(self):
        from paper_2406_18109_gb300 import dist as D
        W = self.W
        cfg = self.cfg = configs.BLACK_SCHOLES
        n = cfg["n"]
        # weak scaling: every rank prices its own, independent batch
        S, K, T = inputs.bs_inputs(n, seed=D.rank_seed(cfg["seed"], int(os.environ.get("RANK", "0"))))
        self.dS, self.dK, self.dT = self.rt.array(S), self.rt.array(K), self.rt.array(T)
        self.units = n
        self.step = self._bs
        if not self.e2e and self.graph_mode:
            # the batch's window (23 tasks, stores into call and put) issued
            # once, then captured once and replayed per step, as a pricing
            # loop over resident data would run it
            rt = self.rt
            self.dcall = rt.empty((n,), np.float32)
            self.dput = rt.empty((n,), np.float32)

            def window():
                W.black_scholes(self.dS, self.dK, self.dT, cfg["r"], cfg["sigma"], out=(self.dcall, self.dput))
                rt.flush()
            window()
            rt.capture_begin()
            window()
            self.graph = rt.capture_end()
            self.kernel_name = kernel_name_of(rt)
            self.step = self._cg_graph
        if not self.e2e:
            return
        # end to end: S, K, T from pinned host memory, call and put back to it
        self.hS, self.hK, self.hT = self._pin(S), self._pin(K), self._pin(T)
        self.hc = self._pin(np.empty(n, np.float32))
        self.hp = self._pin(np.empty(n, np.float32))
        self.h2d, self.d2h = 3 * n * 4, 2 * n * 4
        self.e2e_mode = cfg["e2e_mode"]
        if self.e2e_mode == "zero_copy":
            # the kernel reads S, K, T from and writes call, put to the host
            # buffers themselves (mapped page-locked memory)
            self.wS, self.wK, self.wT = (self.rt.wrap_host(h) for h in (self.hS, self.hK, self.hT))
            self.wc, self.wp = self.rt.wrap_host(self.hc), self.rt.wrap_host(self.hp)
        else:
            # chunks pipelined over several contexts' streams
            from paper_2406_18109_gb300 import pipeline as PL
            self.pipe_rts = PL.pipelined_runtimes(cfg["e2e_contexts"], self.torch.cuda.current_device(),
                                                  **self.rt_kwargs)
            r, sg = cfg["r"], cfg["sigma"]
            self.pipe = PL.ChunkPipeline(self.pipe_rts, lambda S_, K_, T_: W.black_scholes(S_, K_, T_, r, sg),
                                         cfg["e2e_chunk"], [np.float32] * 3)

    def _setup_cg(self):
        A, W, rt = self.A, self.W, self.rt
        cfg = self.cfg = configs.CG
        rp, col, val, xs = inputs.cg_inputs(m=cfg["m"], seed=cfg["seed"])
        self.Am = A.CSR(rt, rp, col, val)
        self.b = self.Am @ rt.array(xs)
        self.units = cfg["iters"]
        self.step = self._cg
        if not self.graph_mode:
            return
        # the whole solve (reset + 50 in-place iterations) captured once after
        # one normally issued window, then replayed per step; iters_per_flush
        # iterations share one window (one launch)
        ipf = cfg.get("iters_per_flush", 1)
        self.s = W.cg_start_inplace(self.b)

        def window():
            for _ in range(ipf):
                W.cg_iteration_inplace(self.Am, self.s)
            rt.flush()
        if self.autotune:
            self._tune(window, {"tile": [256, 432, 512, 864, 1024, 2048], "block": [128, 256, 512], "unroll": [1, 2]},
                       f"cg-{cfg['m']}-{ipf}", 5, "ms_per_window")
        window()
        rt.capture_begin()
        W.cg_reset_inplace(self.s, self.b)
        rt.flush()
        for it in range(cfg["iters"]):
            W.cg_iteration_inplace(self.Am, self.s)
            if (it + 1) % ipf == 0 or it + 1 == cfg["iters"]:
                rt.flush()
        self.graph = rt.capture_end()
        self.kernel_name = kernel_name_of(rt)       # the last iteration window the graph replays
        self.step = self._cg_graph
        if self.e2e:
            # end to end: b uploaded from pinned host memory, x read back, every step
            self.hb = self._pin(self.b.numpy())
            self.hx = self._pin(np.empty(self.hb.shape, self.hb.dtype))
            self.h2d = self.d2h = self.hb.nbytes
            self.e2e_io = ([(self.b, self.hb)], [(self.s.x, self.hx)])

    def _setup_batched(self):
        A, W, rt = self.A, self.W, self.rt
        cfg = self.cfg = configs.BATCHED_CG
        dt = np.float64 if cfg["dtype"] == "f64" else np.float32
        self.probs, self.nnz, self.rows = [], 0, 0
        mats = []
        for spec in inputs.batched_cg_problems(cfg["count"], cfg["seed"]):
            rp, col, val, xs = inputs.batched_cg_matrix(spec)
            mats.append((A.CSR(rt, rp, col, val.astype(dt)), rt.array(xs.astype(dt))))
            self.nnz += len(col)
            self.rows += len(rp) - 1
        # b = A x* and the CG start of every problem, as one batch
        rt.batch_begin()
        for Am, xs_d in mats:
            b = Am @ xs_d
            self.probs.append((Am, W.cg_start_inplace(b), b))
            rt.batch_next()
        rt.batch_end()
        del mats
        pairs = [(Am, s) for Am, s, _ in self.probs]

        def one_iteration():
            if self.per_solve:
                for Am, s in pairs:
                    W.cg_iteration_inplace(Am, s)
                    rt.flush()
            else:
                W.batched_cg_iteration(rt, pairs)

        def reset():
            if self.per_solve:
                for _, s, b in self.probs:
                    W.cg_reset_inplace(s, b)
                    rt.flush()
            else:
                rt.batch_begin()
                for _, s, b in self.probs:
                    W.cg_reset_inplace(s, b)
                    rt.batch_next()
                rt.batch_end()
        if self.autotune:
            # tile cap and launch shape of the batched iteration (coordinate descent)
            self._tune(one_iteration, {"tile_max": [512, 1024, 2048, 4096, 8192], "block": [128, 256, 512],
                                       "unroll": [1, 2], "ctas_per_sm": [0, 5, 6]},
                       f"batched-cg-{cfg['count']}-{cfg['seed']}-{cfg['dtype']}", 3, "ms_per_iteration")
        # one normal pass of each window (compiles kernels, uploads descriptors), then capture
        reset()
        one_iteration()
        rt.capture_begin()
        reset()
        for _ in range(cfg["iters"]):
            one_iteration()
        self.graph = rt.capture_end()
        self.kernel_name = kernel_name_of(rt)       # the last batched iteration the graph replays
        self.units = cfg["count"] * cfg["iters"]
        self.step = self._cg_graph
        if self.e2e:
            ups, downs = [], []
            for _, s, b in self.probs:
                hb = self._pin(b.numpy())
                ups.append((b, hb))
                downs.append((s.x, self._pin(np.empty(hb.shape, hb.dtype))))
            self.h2d = sum(h.nbytes for _, h in ups)
            self.d2h = sum(h.nbytes for _, h in downs)
            self.e2e_io = (ups, downs)

    def _setup_jacobi(self):
        W, rt = self.W, self.rt
        cfg = self.cfg = configs.JACOBI
        grid = inputs.jacobi_grid(cfg["N"], seed=cfg["seed"])
        self.g = rt.array(grid)
        self.views = W.jacobi_views(self.g)
        self.units = cfg["sweeps"]
        self.step = self._jacobi
        if self.autotune:
            # launch shape of the sweep (an in-place sweep depends neither on
            # the rows per point nor on the unroll factor)
            def sweep():
                W.jacobi_sweep(self.views)
                rt.flush()
            self._tune(sweep, {"block": [256, 512], "ctas_per_sm": [0, 2]},
                       f"jacobi-{cfg['N']}", 3, "ms_per_sweep")
        if self.graph_mode:
            # the step's sweeps (one window per sweep, memoised) issued once,
            # then captured once and replayed per step, so no host issue
            # sits between the kernels
            per = cfg["sweeps_per_flush"]

            def window():
                for s in range(cfg["sweeps"]):
                    W.jacobi_sweep(self.views)
                    if (s + 1) % per == 0:
                        rt.flush()
                rt.flush()
            window()
            rt.capture_begin()
            window()
            self.graph = rt.capture_end()
            self.kernel_name = kernel_name_of(rt)
            self.step = self._cg_graph
        if self.e2e:
            hg = self._pin(grid)
            self.h2d = self.d2h = hg.nbytes
            self.e2e_io = ([(self.g, hg)], [(self.g, self._pin(np.empty_like(grid)))])

    # ---------------------------------------------------------------- steps
    def _bs(self):
        c = self.cfg
        if self.e2e and self.e2e_mode == "zero_copy":
            call, put = self.W.black_scholes(self.wS, self.wK, self.wT, c["r"], c["sigma"])
            self.wc[...] = call
            self.wp[...] = put
            del call, put                        # temporaries: the kernel stores into host memory
            self.rt.flush()
            self.rt.sync()
            return
        if self.e2e:
            self.pipe.run([self.hS, self.hK, self.hT], [self.hc, self.hp])
            return
        call, put = self.W.black_scholes(self.dS, self.dK, self.dT, c["r"], c["sigma"])
        self.rt.flush()
        self.keep = (call, put)

    def _cg(self):
        st = self.W.cg_start(self.b)
        self.rt.flush()
        for _ in range(self.cfg["iters"]):
            self.W.cg_iteration(self.Am, st)
            self.rt.flush()
        self.keep = st

    def _cg_graph(self):
        if self.e2e:
            for dev, host in self.e2e_io[0]:
                dev.write(host)
        self.rt.graph_launch(self.graph)
        if self.e2e:
            for dev, host in self.e2e_io[1]:
                dev.read_into(host)

    def _jacobi(self):
        if self.e2e:
            self.g.write(self.e2e_io[0][0][1])
        per = self.cfg["sweeps_per_flush"]
        for s in range(self.cfg["sweeps"]):
            self.W.jacobi_sweep(self.views)
            if (s + 1) % per == 0:
                self.rt.flush()
        self.rt.flush()
        if self.e2e:
            self.g.read_into(self.e2e_io[1][0][1])

    def run(self, steps, warmup):
        torch, stream, rt = self.torch, self.stream, self.rt
        for _ in range(warmup):
            self.step()
        rt.sync()
        s0 = rt.stats()
        torch.cuda.synchronize()
        # an event at every step boundary: the whole region and each step
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
        ev[0].record(stream)
        t0 = time.perf_counter()
        for k in range(steps):
            self.step()
            ev[k + 1].record(stream)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        rt.sync()
        s1 = rt.stats()
        ms = ev[0].elapsed_time(ev[-1])
        per = sorted(ev[k].elapsed_time(ev[k + 1]) for k in range(steps))
        trimmed = per[1:-1] if len(per) > 2 else per
        kd = kernel_delta(s0["kernel_times"], s1["kernel_times"])
        dom = max(kd.items(), key=lambda kv: kv[1]["ms"]) if kd else (None, {"ms": 0.0, "launches": 1})
        out = {"ms": ms, "wall_s": wall, "launches": s1["launches"] - s0["launches"],
               "step_ms": {"p50": statistics.median(per), "min": per[0], "max": per[-1],
                           "trimmed_mean": sum(trimmed) / len(trimmed)},
               "units": self.units * steps, "kernels": kd, "dominant": dom[0],
               "dominant_ms": dom[1]["ms"] / max(1, dom[1]["launches"]),
               "dominant_launches": dom[1]["launches"], "stats": s1}
        return out

    def close(self):
        self.keep = None
        self.pipe = None
        for r in getattr(self, "pipe_rts", []):
            r.close()
        self.rt.close()


def compile_report(torch, stream, sms) -> dict:
    """Warm-up cost of compilation (Section 7.2, Fig. 13): first step (which
    compiles every kernel with NVRTC, no on-disk cache) and steady-state step,
    unfused vs fused, and the steps needed for fusion to pay for compiling."""
    from paper_2406_18109_gb300 import arrays as A
    # NVRTC's one-time start-up (loading its builtins) is paid here, by a
    # kernel none of the measured windows uses
    with A.Runtime(device=torch.cuda.current_device(), stream=stream.cuda_stream) as rt:
        (A.full(rt, (1000,), 1.0) * 3.0).numpy()
    out = {}
    for wl in ("bs", "cg", "jacobi"):
        cfg = {"bs": configs.BLACK_SCHOLES, "cg": configs.CG, "jacobi": configs.JACOBI}[wl]
        base = dict(block=cfg["block"], unroll=cfg["unroll"], sms=sms)
        for k in ("tile", "rows"):
            if k in cfg:
                base[k] = cfg[k]
        row = {}
        for name, kw in (("standard", dict(fusion=False, launch="per_task")),
                         ("compiled", dict(fusion=True, launch="persistent"))):
            a = Arm(wl, dict(base, **kw), torch, stream)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            a.step()
            a.rt.sync()
            first = time.perf_counter() - t0
            r = a.run(3, 1)
            st = a.rt.stats()
            a.close()
            row[name] = {"first_step_s": first, "steady_step_s": r["ms"] / 3 / 1e3,
                         "compile_s": st.get("compile_s"), "kernels": st.get("kernels_compiled")}
        s, c = row["standard"], row["compiled"]
        gain = s["steady_step_s"] - c["steady_step_s"]
        extra = c["first_step_s"] - s["first_step_s"]
        row["breakeven_steps"] = (extra / gain) if (extra > 0 and gain > 0) else None
        row["step"] = {"bs": "one 2^26-option batch", "cg": "one 50-iteration solve",
                       "jacobi": "200 sweeps"}[wl]
        out[wl] = row
    return out


def serving_alg_bytes(results) -> int:
    """Algorithmic HBM bytes of the served work: per solver iteration the CSR
    matrix once per SpMV (12 B per entry, 4 B per row pointer) plus the vector
    passes the phases need (CG 88 B per row; BiCGSTAB 168 B per row, two SpMVs),
    per option batch 20 B per option."""
    from paper_2406_18109_gb300 import serve as SV
    tot = 0
    for r in results:
        if r.kind == "bs":
            tot += 20 * r.size
            continue
        n = r.size ** 3
        mat = SV.operator_bytes(r.size)
        per = mat + 88 * n if r.kind == "cg" else 2 * mat + 168 * n
        tot += r.iterations * per
    return tot


def run_serving(args, env):
    """The serving loop under its Poisson arrival stream, then again at a
    fraction of the throughput it sustained; one JSON line.  With N GPUs every
    rank serves its own stream (replicas; seeds differ by rank) and the value
    is the requests of all ranks over the slowest rank's time."""
    from paper_2406_18109_gb300 import arrays as A
    from paper_2406_18109_gb300 import dist as D
    from paper_2406_18109_gb300 import serve as SV
    torch, stream, sms, cache, dev = env["torch"], env["stream"], env["sms"], env["cache"], env["dev"]
    cfg = configs.SERVING
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    seed = D.rank_seed(cfg["seed"], rank)
    count = args.requests or cfg["count"]
    peaks = load_peaks()
    # command-line overrides of the launch shape (tuning), as for the other workloads
    shape = {k: getattr(args, k) or cfg[k] for k in ("tile", "block", "unroll")}
    rt = A.Runtime(device=dev, stream=stream.cuda_stream, time_launches=True, tile=shape["tile"],
                   block=shape["block"], unroll=shape["unroll"], sms=sms, cache_dir=cache)

    def server():
        return SV.Server(rt, inputs.poisson3d_csr, budget_bytes=int(cfg["budget_gb"] * 1e9), tol=cfg["tol"],
                         iters_per_tick=cfg["iters_per_tick"], max_active=cfg["max_active"], keep_outputs=False,
                         overlap=not args.no_overlap, templates=not args.no_templates)

    # resident operators (every rung of the ladder), loaded before serving
    t_load = time.perf_counter()
    srv = server()
    for m in inputs.SERVE_LADDER:
        srv._operator(m)
    rt.sync()
    t_load = time.perf_counter() - t_load
    # warm-up: compile the kernels of every window shape on a few requests
    warm = inputs.serving_requests(12, seed=99, mean_gap_s=1e-4, ladder=inputs.SERVE_LADDER[:2], bs_log2=(16, 17))
    srv.run(warm, inputs.serving_payload)

    def one_run(mean_gap_s):
        reqs = inputs.serving_requests(count, seed=seed, mean_gap_s=mean_gap_s)
        # request data arrive with the requests, in mapped page-locked host
        # buffers the server reads in place: generated (in parallel, the
        # generators release the GIL) before the clock starts
        import concurrent.futures as cf

        def pinned(req):
            p = inputs.serving_payload(req)
            out = []
            for a in (p if isinstance(p, tuple) else (p,)):
                h = A.Runtime.host_empty(a.shape, a.dtype)
                h[...] = a
                out.append(h)
            return tuple(out) if isinstance(p, tuple) else out[0]
        with cf.ThreadPoolExecutor(8) as ex:
            data = dict(zip([r["rid"] for r in reqs], ex.map(pinned, reqs)))
        rt.sync()
        s0 = rt.stats()
        h0 = dict(srv.stats.host_s)
        clocks = Clocks(dev)
        clocks.start()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        res = srv.run(reqs, lambda r: data.pop(r["rid"]))
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        clk = clocks.stop()
        rt.sync()
        s1 = rt.stats()
        kd = kernel_delta(s0["kernel_times"], s1["kernel_times"])
        kern_ms = sum(v["ms"] for v in kd.values())
        summ = SV.summarize(res, wall)
        alg = serving_alg_bytes(res)
        summ.update({"offered_rps": 1.0 / mean_gap_s, "mean_gap_ms": mean_gap_s * 1e3,
                     "kernel_ms": kern_ms, "gpu_busy_frac": kern_ms / 1e3 / wall if wall > 0 else 0.0,
                     "algorithmic_bytes": alg, "launches": s1["launches"] - s0["launches"],
                     "batched_launches": s1["batches"] - s0["batches"],
                     "repeated_launches": s1["batch_repeats"] - s0["batch_repeats"],
                     "h2d_bytes": sum(r.size ** 3 * 8 if r.kind != "bs" else 12 * r.size for r in res),
                     "d2h_bytes": sum(r.size ** 3 * 8 if r.kind != "bs" else 8 * r.size for r in res),
                     "peak_device_bytes": srv.stats.peak_bytes, "max_active": dict(srv.stats.max_active)})
        top = max(kd.items(), key=lambda kv: kv[1]["ms"]) if kd else (None, {"ms": 0.0, "launches": 0})
        summ["dominant_kernel"] = {"name": top[0], "ms": top[1]["ms"], "launches": top[1]["launches"]}
        summ["result_buffers"] = dict(srv.stats_pool)
        summ["host_s_by_part"] = {k: v - h0.get(k, 0.0) for k, v in srv.stats.host_s.items()}
        return summ, clk

    if world > 1:
        torch.distributed.barrier()
    offered, clk = one_run(cfg["mean_gap_ms"] * 1e-3)
    if world > 1:
        # whole-job throughput: every rank's requests over the slowest rank's time
        v, ms, _ = D.combine(offered["wall_s"] * 1e3, offered["requests"], device="cuda")
        offered["sustained_rps_all_ranks"] = v
    cap = offered["sustained_rps"]
    at_load = None
    if not args.quick and cap > 0:
        at_load, _ = one_run(1.0 / (cfg["load_fraction"] * cap))
    achieved = offered["algorithmic_bytes"] / (offered["kernel_ms"] / 1e3) / 1e9 if offered["kernel_ms"] > 0 else 0.0
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                "frac": achieved / peaks["hbm_gbs"], "traffic": None, "peak_source": peaks["source"],
                "kernel": "all kernels of the run (batched CG/BiCGSTAB iterations dominate)",
                "kernel_ms": offered["kernel_ms"], "launches": offered["launches"],
                "algorithmic_bytes_per_launch": offered["algorithmic_bytes"] / max(1, offered["launches"])}
    cpu = None
    if not args.quick and rank == 0:
        v, u, sample = oracle_rate("serve", budget_s=10.0)
        cpu = {"value": v, "unit": u, "cores": 1, "kind": "oracle", "sample": sample}
    n = offered["requests"]
    value = offered.get("sustained_rps_all_ranks", offered["sustained_rps"])
    line = {"metric": METRIC["serve"][0], "value": value, "unit": "requests/s", "n_gpus": world,
            "steps": n, "warmup": len(warm), "ms_per_step": offered["wall_s"] * 1e3 / max(1, n),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64+f32",
            "data": "synthetic (seeded generators of synth/inputs.py)",
            "config": {"workload": WORKLOAD["serve"], "requests": n, "l2": "inputs larger than L2",
                       "launch": "continuous batching: one batched persistent launch per solver kind per "
                                 "iteration, dfs_batch_repeat within a tick",
                       "parallelism": f"replicas x{world}", "shape": shape},
            "p50_ms": offered["p50_ms"], "p99_ms": offered["p99_ms"],
            "e2e": {"value": value, "unit": "requests/s",
                    "h2d_bytes_per_step": offered["h2d_bytes"] / max(1, n),
                    "d2h_bytes_per_step": offered["d2h_bytes"] / max(1, n),
                    "note": "a step is one request; payload upload and result download are inside the loop"},
            "gpu_launches": offered["launches"], "roofline": roofline, "cpu_baseline": cpu, "clocks": clk,
            "serving": {"offered_load": offered, "at_fraction_of_capacity": at_load,
                        "load_fraction": cfg["load_fraction"], "operator_load_s": t_load}}
    rt.close()
    return line


def measure(args, workload, env, steps, warmup, cpu_budget=(10.0, 8.0)) -> dict:
    """Times one workload (fused persistent arm, then the comparison arms, the
    end-to-end arm and the CPU oracle) and returns its JSON line.  env holds
    the device plumbing: torch, stream, sms, cache, dev, world, rank."""
    torch, stream, sms, cache = env["torch"], env["stream"], env["sms"], env["cache"]
    dev, world, rank = env["dev"], env["world"], env["rank"]
    from paper_2406_18109_gb300 import dist as D
    metric, unit, dtype = METRIC[workload]
    cfg = {"bs": configs.BLACK_SCHOLES, "cg": configs.CG, "jacobi": configs.JACOBI,
           "batched": configs.BATCHED_CG}[workload]
    base = dict(block=cfg["block"], unroll=cfg["unroll"], sms=sms, cache_dir=cache)
    for k in ("tile", "tile_max", "min_points", "window_size"):
        if k in cfg:
            base[k] = cfg[k]
    if "rows" in cfg:
        base["rows"] = cfg["rows"]
    for k in ("block", "unroll", "tile", "rows"):       # command-line overrides (tuning)
        if getattr(args, k):
            base[k] = getattr(args, k)
    if "ctas_per_sm" in cfg:
        base["ctas_per_sm"] = cfg["ctas_per_sm"]
    if args.ctas >= 0:
        base["ctas_per_sm"] = args.ctas
    if "stage_x" in cfg:
        base["stage_x"] = cfg["stage_x"]
    if args.stage_x:
        base["stage_x"] = args.stage_x == "on"

    # CG: the iteration windows are captured once (memoised windows + a CUDA
    # graph) and replayed; the Python-issued runs are reported beside them
    graph = workload in ("cg", "batched", "bs", "jacobi")

    def arm(kw, steps, warmup, e2e=False, graph=graph, per_solve=False):
        a = Arm(workload, kw, torch, stream, e2e=e2e, graph=graph, per_solve=per_solve)
        try:
            return a.run(steps, warmup)
        finally:
            a.close()

    fused_arm = Arm(workload, dict(base, fusion=True, launch="persistent"), torch, stream, graph=graph,
                    autotune=workload in ("batched", "jacobi", "cg") and not args.no_autotune)
    batch_sizes = (fused_arm.nnz, fused_arm.rows) if workload == "batched" else None
    tuned = fused_arm.tuned
    if tuned:
        # the comparison arms run with the tuned setting too
        base.update(tuned["config"])
    clocks = Clocks(dev)
    if world > 1:
        torch.distributed.barrier()
    clocks.start()
    time.sleep(1.0)                              # let the clock sampler start before timing
    fused = fused_arm.run(steps, warmup)
    clk = clocks.stop()
    fused_arm.close()
    value, fused["ms"], _ = D.combine(fused["ms"], fused["units"], device="cuda" if world > 1 else None)
    ms_step = fused["ms"] / steps

    extra = {}
    if not args.quick and workload == "batched":
        k2 = max(2, steps // 2)
        ps = arm(dict(base, fusion=True, launch="persistent"), k2, 1, per_solve=True)
        extra["per_solve_launches"] = {"value": ps["units"] / (ps["ms"] / 1e3), "ms_per_step": ps["ms"] / k2,
                                       "note": "same fused windows, one launch per solve per iteration, "
                                               "replayed from a CUDA graph"}
        extra["batched_vs_per_solve"] = value / world / extra["per_solve_launches"]["value"]
    elif not args.quick:
        k2 = max(3, steps // 4)
        unf = arm(dict(base, fusion=False, launch="per_task"), k2, 2)
        pt = arm(dict(base, fusion=True, launch="per_task"), k2, 2)
        def kms(run, k):
            # summed per-launch device times; launches replayed from a graph
            # are not timed one by one (null then)
            t = sum(v["ms"] for v in run["kernels"].values())
            return t / k if t > 0 else None
        extra["unfused"] = {"value": unf["units"] / (unf["ms"] / 1e3), "ms_per_step": unf["ms"] / k2,
                            "launches_per_step": unf["launches"] / k2, "kernel_ms_per_step": kms(unf, k2)}
        extra["fused_per_task"] = {"value": pt["units"] / (pt["ms"] / 1e3), "ms_per_step": pt["ms"] / k2,
                                   "launches_per_step": pt["launches"] / k2, "kernel_ms_per_step": kms(pt, k2)}
        extra["fused_vs_unfused"] = value / world / extra["unfused"]["value"]
        extra["fused_kernel_ms_per_step"] = kms(fused, steps)
        if graph:
            nf = arm(dict(base, fusion=True, launch="persistent"), k2, 2, graph=False)
            nu = arm(dict(base, fusion=False, launch="per_task"), k2, 2, graph=False)
            extra["python_issued"] = {
                "fused": {"value": nf["units"] / (nf["ms"] / 1e3), "ms_per_step": nf["ms"] / k2},
                "unfused": {"value": nu["units"] / (nu["ms"] / 1e3), "ms_per_step": nu["ms"] / k2},
                "note": {"bs": "each batch issued from Python (23 tasks + flush)",
                         "jacobi": "each sweep issued from Python (6 tasks + flush)"}.get(
                             workload, "each iteration issued from Python (11 tasks + flush); host-bound")}
    if not args.quick:
        # end to end through the public API: inputs from pinned host memory
        # and results back to it inside every timed step
        k3 = max(2, steps // 4)
        ea = Arm(workload, dict(base, fusion=True, launch="persistent"), torch, stream, e2e=True, graph=graph)
        try:
            e = ea.run(k3, 2)
            extra["e2e"] = {"value": e["units"] / (e["ms"] / 1e3), "unit": unit,
                            "h2d_bytes_per_step": ea.h2d, "d2h_bytes_per_step": ea.d2h}
            # the host link as a roofline of the end-to-end step: bytes that
            # cross it per step over the step time, against copies both ways
            # at once, measured now
            link = host_link_peak(torch)
            moved = (ea.h2d + ea.d2h) / (e["ms"] / 1e3 / k3) / 1e9
            extra["e2e"]["roofline"] = {"bound": "host link", "achieved": moved, "peak": link["both"], "unit": "GB/s",
                                        "frac": moved / link["both"], "peak_source": "measured: pinned copies both ways "
                                        "at once (h2d %.0f, d2h %.0f GB/s alone)" % (link["h2d"], link["d2h"])}
        finally:
            ea.close()

    peaks = load_peaks()
    if workload == "bs":
        alg_bytes = 20 * cfg["n"]                          # read S, K, T; write call, put
    elif workload == "cg":
        m = cfg["m"]
        nn, nnz = m * m, 5 * m * m - 4 * m
        alg_bytes = 12 * nnz + 4 * (nn + 1) + 96 * nn     # one CG iteration
    elif workload == "batched":
        nnz, rows = batch_sizes
        esz = 8 if cfg["dtype"] == "f64" else 4
        # per batched iteration, summed over the solves: CSR (value + int32
        # column per entry, int32 row pointers) and the vector passes of the
        # iteration (12 for the FP64 count of the single-solve CG line)
        alg_bytes = (esz + 4) * nnz + 4 * (rows + cfg["count"]) + 12 * esz * rows
    else:
        # one sweep (one launch), in place: every point read once and written
        # once (the two phases of before moved twice that)
        alg_bytes = 8 * cfg["N"] * cfg["N"]
    kern_ms = fused["dominant_ms"]
    if graph:
        # launches replayed from a graph are not timed one by one: use the
        # replayed time per iteration (kernel plus the gap to the next node)
        its = cfg.get("iters", cfg.get("sweeps", 1))
        kern_ms = fused["ms"] / (steps * its)
        fused["dominant"] = {"batched": "batched CG iteration kernel", "cg": "CG iteration kernel",
                             "bs": "fused Black-Scholes kernel", "jacobi": "Jacobi sweep kernel"}[workload] + \
            ", graph replay (time per launch incl. the gap to the next)"
        fused["dominant_launches"] = steps * its
    achieved = alg_bytes / (kern_ms / 1e3) / 1e9 if kern_ms > 0 else 0.0
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                "frac": achieved / peaks["hbm_gbs"], "traffic": None,
                "peak_source": peaks["source"], "kernel": fused["dominant"], "kernel_ms": kern_ms,
                "launches": fused["dominant_launches"], "algorithmic_bytes_per_launch": alg_bytes}
    # measured DRAM traffic (ncu) of the dominant kernel, used only when the
    # kernel timed now is the one the counters were taken on (same generated
    # code, so the same name) at the default size; else null
    kname = fused_arm.kernel_name if graph else fused["dominant"]
    ctr = counters_for(cfg, kname)
    roofline["kernel_name"] = kname
    roofline["counters_kernel"] = counters_kernels(cfg)
    if ctr and workload == "cg" and cfg["m"] == 256:
        roofline["traffic"] = ctr["dram_bytes_per_iteration"]
    elif ctr and workload == "batched" and cfg["count"] == 256:
        roofline["traffic"] = ctr["dram_bytes_per_launch"]
    elif ctr and workload == "jacobi" and cfg["N"] == 8190:
        roofline["traffic"] = ctr["dram_bytes_per_launch"]
    fp64_ops = None
    if workload == "cg":
        fp64_ops = nnz + 8 * nn
    elif workload == "batched" and cfg["dtype"] == "f64":
        fp64_ops = nnz + 8 * rows
    if fp64_ops is not None:
        # FP64 is a scarce pipe on GB300 (nominal 1.25 TFLOP/s counting an FMA
        # as two: about two lane operations per SM and clock).  Lane operations
        # per iteration: one FMA per stored entry (SpMV) and eight per row (the
        # two dots, the x, r and p updates at two operations each but the dots'
        # one)
        sm_max = clk.get("sm_max_mhz") or 2070.0
        peak_ops = sms * 2 * sm_max * 1e6 / 1e9
        ach_ops = fp64_ops / (kern_ms / 1e3) / 1e9 if kern_ms > 0 else 0.0
        roofline["fp64"] = {"achieved": ach_ops, "peak": peak_ops, "unit": "G lane-ops/s", "frac": ach_ops / peak_ops,
                            "ops_per_launch": fp64_ops,
                            "peak_source": f"derived: {sms} SMs x 2 FP64 lanes x {sm_max:.0f} MHz (1.25 TFLOP/s nominal)"}
    if workload == "bs":
        # issue-bound: instructions per option (ncu) x options / kernel time,
        # against SMs x 4 sub-partitions x 32 lanes x maximum SM clock
        sm_max = clk.get("sm_max_mhz") or 2070.0
        peak_ti = sms * 4 * 32 * sm_max * 1e6 / 1e12
        # the instruction count and DRAM traffic (ncu) belong to one generated
        # kernel: used only when that kernel is the one timed now, else null
        ctr = counters_for(cfg, fused_arm.kernel_name or fused["dominant"]) if cfg["n"] == 1 << 26 else None
        hbm = {"achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s", "frac": achieved / peaks["hbm_gbs"],
               "peak_source": peaks["source"], "algorithmic_bytes_per_launch": alg_bytes}
        if ctr:
            ach_ti = ctr["inst_per_option"] * cfg["n"] / (kern_ms / 1e3) / 1e12 if kern_ms > 0 else 0.0
            roofline = {"bound": "alu", "achieved": ach_ti, "peak": peak_ti, "unit": "T thread-inst/s",
                        "frac": ach_ti / peak_ti, "traffic": ctr["dram_bytes_per_launch"],
                        "peak_source": f"derived: {sms} SMs x 4 SMSPs x 32 lanes x {sm_max:.0f} MHz",
                        "inst_per_option": ctr["inst_per_option"], "hbm": hbm}
        else:
            roofline = dict(hbm, bound="hbm", traffic=None, inst_per_option=None)
        roofline.update({"kernel": fused["dominant"], "kernel_name": fused_arm.kernel_name or fused["dominant"],
                         "counters_kernel": counters_kernels(cfg), "kernel_ms": kern_ms,
                         "launches": fused["dominant_launches"]})

    cpu = None
    if rank == 0 and world == 1 and not args.quick:
        v, u, sample = oracle_rate(workload, budget_s=cpu_budget[0])
        cpu = {"value": v, "unit": u, "cores": 1, "kind": "oracle", "sample": sample}
        if workload in ALL_CORES_SAMPLE:
            va, nc = oracle_rate_all_cores(workload, cpu_budget[1])
            cpu["all_cores"] = {"value": va, "unit": u, "cores": nc,
                                "sample": ALL_CORES_SAMPLE[workload] + f", {cpu_budget[1]:.0f} s"}

    line = {"metric": metric, "value": value, "unit": unit, "n_gpus": world, "steps": steps,
            "warmup": warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": dtype, "data": "synthetic (seeded generators of synth/inputs.py)",
            "config": {"workload": WORKLOAD[workload],
                       "l2": "inputs larger than L2" if workload != "cg"
                       else "working set L2-resident (10 MB); no flush",
                       "launch": "persistent fused" + ((", each batch replayed from a CUDA graph of the memoised "
                                                         "window" if workload == "bs" else
                                                         ", each step's sweeps replayed from a CUDA graph of the "
                                                         "memoised sweep windows" if workload == "jacobi" else
                                                         ", each solve replayed from a CUDA graph of the memoised "
                                                         "iteration windows") if graph else ""),
                       "parallelism": f"replicas x{world}"},
            "e2e": extra.pop("e2e", None), "gpu_launches": fused["launches"], "roofline": roofline,
            "step_ms": fused["step_ms"],
            "cpu_baseline": cpu, "clocks": clk}
    line.update(extra)
    if tuned:
        line["config"]["autotuned"] = tuned["config"]
        line["autotune"] = tuned["trials"]
    st = fused["stats"]
    line["runtime_stats"] = {k: st.get(k) for k in ("compile_s", "kernels_compiled", "plan_hits", "plan_misses",
                                                     "kernel_disk_hits", "last_regs", "last_occupancy",
                                                     "last_grid", "last_block", "analysis_s")}
    return line


def counters_for(cfg: dict, kernel_name):
    """The ncu counters stored for a workload, if they were taken on the kernel
    named (its name hashes its generated body), else None."""
    ctrs = cfg.get("counters") or []
    for ctr in ([ctrs] if isinstance(ctrs, dict) else ctrs):
        if kernel_name and ctr.get("kernel") == kernel_name:
            return ctr
    return None


def counters_kernels(cfg: dict):
    """Names of the kernels a workload's stored counters belong to."""
    ctrs = cfg.get("counters") or []
    return [c["kernel"] for c in ([ctrs] if isinstance(ctrs, dict) else ctrs)]


COMPACT_KEYS = ("metric", "value", "unit", "steps", "warmup", "ms_per_step", "dtype", "config", "gpu_launches",
                "roofline", "e2e", "cpu_baseline", "clocks", "step_ms", "fused_vs_unfused", "unfused", "fused_per_task",
                "fused_kernel_ms_per_step", "python_issued", "batched_vs_per_solve", "per_solve_launches")


def compact(line: dict) -> dict:
    """A workload's line as a sub-object of the default line (its own value,
    timing, comparison arms, roofline and oracle rate; the tuner's trial list
    and the runtime counters left out)."""
    return {k: line[k] for k in COMPACT_KEYS if k in line}


def compact_serving(line: dict) -> dict:
    """The serving line as a sub-object: sustained requests/s under the
    offered Poisson load, and p50/p99 latency both there and at the stated
    fraction of that throughput."""
    out = {k: line[k] for k in ("metric", "value", "unit", "p50_ms", "p99_ms", "dtype", "config", "gpu_launches",
                                "roofline", "e2e", "cpu_baseline", "clocks") if k in line}
    srv = line["serving"]
    off = srv["offered_load"]
    out["offered_load"] = {k: off.get(k) for k in ("offered_rps", "sustained_rps", "p50_ms", "p99_ms", "requests",
                                                    "wall_s", "gpu_busy_frac", "unconverged")}
    at = srv.get("at_fraction_of_capacity")
    if at:
        out["at_fraction_of_capacity"] = {"load_fraction": srv["load_fraction"],
                                          **{k: at.get(k) for k in ("offered_rps", "sustained_rps", "p50_ms", "p99_ms",
                                                                    "requests", "wall_s", "gpu_busy_frac",
                                                                    "unconverged")}}
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=0,
                    help="timed steps (default 50 for the sub-millisecond Black-Scholes step, else 20)")
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="bs", choices=["bs", "cg", "jacobi", "batched", "serve"])
    ap.add_argument("--requests", type=int, default=0, help="serving: requests per run (default: the config's)")
    ap.add_argument("--no-templates", action="store_true",
                    help="serving: issue every iteration task by task instead of replaying recorded windows")
    ap.add_argument("--no-overlap", action="store_true",
                    help="serving: one group of solves (the host waits for every convergence read)")
    ap.add_argument("--fp32", action="store_true", help="batched CG in FP32 instead of FP64")
    ap.add_argument("--quick", action="store_true", help="skip the comparison arms (for profiling)")
    ap.add_argument("--no-extras", action="store_true",
                    help="Black-Scholes line only (no CG, Jacobi and serving sub-objects)")
    ap.add_argument("--bs-n", type=int, default=0, help="Black-Scholes batch size (profiling a smaller case)")
    ap.add_argument("--jac-n", type=int, default=0, help="Jacobi interior size N (profiling a smaller case)")
    ap.add_argument("--sweeps", type=int, default=0, help="Jacobi sweeps per step (profiling)")
    for k in ("block", "unroll", "tile", "rows"):
        ap.add_argument(f"--{k}", type=int, default=0, help=f"override the workload's {k} (tuning)")
    ap.add_argument("--ipf", type=int, default=0, help="CG: iterations per flush window (tuning)")
    ap.add_argument("--ctas", type=int, default=-1, help="resident CTAs per SM to size for (tuning; 0 = as many as fit)")
    ap.add_argument("--e2e-chunk", type=int, default=0, help="Black-Scholes end to end: options per chunk (tuning)")
    ap.add_argument("--e2e-contexts", type=int, default=0, help="Black-Scholes end to end: streams (tuning)")
    ap.add_argument("--e2e-mode", default="", choices=["", "zero_copy", "pipeline"],
                    help="Black-Scholes end to end: kernels on mapped host memory, or pipelined copies")
    ap.add_argument("--stage-x", default="", choices=["", "on", "off"],
                    help="SpMV x windows staged in shared memory (default: the workload's configuration)")
    ap.add_argument("--no-autotune", action="store_true",
                    help="CG / batched CG / Jacobi: keep the configured tiling and launch shape")
    ap.add_argument("--compile-report", action="store_true",
                    help="print the warm-up/compilation cost table instead of the bench line")
    args = ap.parse_args()
    if not args.steps:
        args.steps = 50 if args.workload == "bs" else 20
    if args.bs_n:
        configs.BLACK_SCHOLES["n"] = args.bs_n
    if args.jac_n:
        configs.JACOBI["N"] = args.jac_n
    if args.sweeps:
        configs.JACOBI["sweeps"] = args.sweeps
    if args.ipf:
        configs.CG["iters_per_flush"] = args.ipf
    if args.e2e_chunk:
        configs.BLACK_SCHOLES["e2e_chunk"] = args.e2e_chunk
    if args.e2e_contexts:
        configs.BLACK_SCHOLES["e2e_contexts"] = args.e2e_contexts
    if args.e2e_mode:
        configs.BLACK_SCHOLES["e2e_mode"] = args.e2e_mode
    if args.fp32:
        configs.BATCHED_CG["dtype"] = "f32"
        METRIC["batched"] = (METRIC["batched"][0], "iterations/s", "f32")
        WORKLOAD["batched"] = "batched-cg-256-uneven-100it-fp32"
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    metric, unit, dtype = METRIC[args.workload]

    if args.impl == "reference":
        if rank != 0:
            return
        v, u, sample = oracle_rate(args.workload, budget_s=max(5.0, min(30.0, 2.0 * args.steps)))
        line = {"metric": metric, "value": v, "unit": unit, "n_gpus": args.gpus, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": None, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": dtype, "data": "synthetic", "impl": "reference",
                "config": {"workload": WORKLOAD[args.workload]},
                "cpu_baseline": {"value": v, "unit": u, "cores": 1, "kind": "oracle", "sample": sample},
                "e2e": {"value": v, "unit": u, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line))
        return

    import torch
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
        torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    else:
        torch.cuda.set_device(0)
    dev = torch.cuda.current_device()
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    # compiled kernels are kept on disk between runs (Section 7.2's suggested follow-up)
    import tempfile
    cache = os.path.join(tempfile.gettempdir(), "dfs_cubins")
    os.makedirs(cache, exist_ok=True)

    from paper_2406_18109_gb300 import _build
    _build.build()
    if args.compile_report:
        print(json.dumps({"compile_report": compile_report(torch, stream, sms)}))
        return
    env = dict(torch=torch, stream=stream, sms=sms, cache=cache, dev=dev, world=world, rank=rank)
    if args.workload == "serve":
        line = run_serving(args, env)
    else:
        line = measure(args, args.workload, env, args.steps, args.warmup)
        if args.workload == "bs" and not args.quick and not args.no_extras:
            # the other half of the headline metric in the same line: CG
            # iterations/s, Jacobi sweeps/s and the serving loop's p50/p99,
            # each with its own fused/unfused ratio, roofline and oracle rate
            line["cg"] = compact(measure(args, "cg", env, 20, 3, cpu_budget=(5.0, 4.0)))
            line["jacobi"] = compact(measure(args, "jacobi", env, 10, 3, cpu_budget=(5.0, 4.0)))
            line["serve"] = compact_serving(run_serving(args, env))
    if rank == 0:
        print(json.dumps(line))
    if world > 1:
        torch.distributed.destroy_process_group()



if __name__ == "__main__":
    main()
