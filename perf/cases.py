"""Measured cases: what a program has the framework do, through its public API.

The programs are the ones this repository serves (workloads.py): Black-Scholes
batches, conjugate gradients (alone and batched), BiCGSTAB ticks of the
serving loop, Jacobi stencils in 2-D and 3-D, and array expressions with
reductions.  Steady loops are captured once and replayed, as the benchmark and
a production loop do; the smallest calls and the array expression are issued
from Python on every pass.  Launch shapes are those of configs.py, or the
Runtime's defaults (a program that sets nothing).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_18109_gb300 import arrays as A
from paper_2406_18109_gb300 import configs
from paper_2406_18109_gb300 import workloads as W

_RATE, _SIGMA = configs.BLACK_SCHOLES["r"], configs.BLACK_SCHOLES["sigma"]
_TORCH = {"f32": torch.float32, "f64": torch.float64}
_NUMPY = {"f32": np.float32, "f64": np.float64}


def listed():
    return [
        # a pricing service's small request: one issue of the 23-task window,
        # where launch and issue latency are everything
        {"name": "bs_4k_issued", "kind": "bs", "n": 4096, "launch": "default", "graph": False},
        # an ordinary odd-sized batch inside a replayed pricing loop
        {"name": "bs_1m_ragged", "kind": "bs", "n": 1000003, "launch": "bs", "graph": True},
        # the full-size batch of the repository's headline workload
        {"name": "bs_64m", "kind": "bs", "n": 1 << 26, "launch": "bs", "graph": True},
        # z = (x - y) / |x - y| with the sum and dot of the inputs: an array
        # expression around reductions, issued as written, odd length
        {"name": "normalise_16m_f32", "kind": "norm", "n": (1 << 24) + 43, "dtype": "f32"},
        # one L2-resident FP64 solve of 50 iterations, five per window
        {"name": "cg_256", "kind": "cg", "m": 256, "iters": 50, "per_flush": 5, "launch": "cg"},
        # a solve larger than L2, odd grid, default launch shape
        {"name": "cg_1337", "kind": "cg", "m": 1337, "iters": 10, "per_flush": 1, "launch": "default"},
        # many uneven solves (2-D Poisson and random SPD), one launch per iteration
        {"name": "batched_cg_f64", "kind": "batched", "count": 96, "mix": 4, "mmax": 1024, "nmax": 65536,
         "iters": 6, "dtype": "f64"},
        {"name": "batched_cg_f32", "kind": "batched", "count": 64, "mix": 7, "mmax": 1024, "nmax": 65536,
         "iters": 6, "dtype": "f32"},
        # one tick of the serving loop: 8 BiCGSTAB iterations of the active
        # solves on 3-D 7-point operators of its ladder
        {"name": "bicgstab_tick_3d", "kind": "bicg", "sides": "64,91,108,128", "iters": 8},
        # the Fig. 1 stencil at full size, one window per sweep
        {"name": "jacobi_8190_f32", "kind": "jacobi2d", "rows": 8190, "cols": 8190, "sweeps": 8, "per_flush": 1,
         "dtype": "f32", "launch": "jacobi"},
        # a small odd grid that stays in L2, several sweeps per window
        {"name": "jacobi_1021_f32", "kind": "jacobi2d", "rows": 1021, "cols": 1147, "sweeps": 40, "per_flush": 5,
         "dtype": "f32", "launch": "default"},
        # the 7-point stencil in 3-D, FP64
        {"name": "jacobi3d_251_f64", "kind": "jacobi3d", "m": 251, "sweeps": 8, "per_flush": 1, "dtype": "f64",
         "launch": "default"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bs", "bs", "norm", "cg", "cg", "batched", "bicg", "jacobi2d", "jacobi2d", "jacobi3d"])
    if kind == "bs":
        issued = rng.random() < 0.25
        n = _log(rng, 100, 30000) if issued else _log(rng, 1 << 14, 1 << 26)
        return {"kind": kind, "n": n, "launch": "default" if issued else "bs", "graph": not issued}
    if kind == "norm":
        return {"kind": kind, "n": _log(rng, 1 << 20, 1 << 24), "dtype": rng.choice(["f32", "f64"])}
    if kind == "cg":
        m = _log(rng, 40, 1337)
        per = rng.choice([1, 5]) if m < 600 else 1
        return {"kind": kind, "m": m, "iters": 10, "per_flush": per, "launch": "cg" if per > 1 else "default"}
    if kind == "batched":
        return {"kind": kind, "count": rng.randint(3, 64), "mix": rng.randint(10, 10 ** 6), "mmax": _log(rng, 200, 1024),
                "nmax": _log(rng, 4000, 65536), "iters": rng.randint(2, 6), "dtype": rng.choice(["f32", "f64"])}
    if kind == "bicg":
        sides = [_log(rng, 40, 128) for _ in range(rng.randint(1, 4))]
        return {"kind": kind, "sides": ",".join(str(m) for m in sides), "iters": rng.randint(4, 8)}
    if kind == "jacobi2d":
        r, c = _log(rng, 200, 8190), _log(rng, 200, 8190)
        per = rng.choice([1, 5])
        return {"kind": kind, "rows": r, "cols": c, "sweeps": rng.randint(1, 3) * 5 if per == 5 else rng.randint(3, 8),
                "per_flush": per, "dtype": rng.choice(["f32", "f32", "f64"]) if r * c < 1 << 25 else "f32",
                "launch": rng.choice(["jacobi", "default"])}
    return {"kind": kind, "m": _log(rng, 40, 251), "sweeps": rng.randint(3, 8), "per_flush": rng.choice([1, 2]),
            "dtype": rng.choice(["f32", "f64"]), "launch": "default"}


# ------------------------------------------------------------------ plumbing
_runtimes = {}


def _runtime(launch):
    """One context per launch shape, kept for the life of the program."""
    if launch not in _runtimes:
        pick = {"default": ({}, ()), "bs": (configs.BLACK_SCHOLES, ("tile", "block", "unroll")),
                "cg": (configs.CG, ("tile", "block", "unroll", "window_size")),
                "jacobi": (configs.JACOBI, ("rows", "block", "unroll")),
                "batched": (configs.BATCHED_CG, ("tile_max", "min_points", "block", "unroll")),
                "serve": (configs.SERVING, ("tile", "block", "unroll"))}[launch]
        _runtimes[launch] = A.Runtime(**{k: pick[0][k] for k in pick[1]})
    return _runtimes[launch]


class _Memory:
    """A store's device memory as other CUDA code sees it (rows of 2-D and 3-D
    stores are pitched to 16 bytes)."""

    def __init__(self, a):
        self.array = a
        item = a.dtype.itemsize
        pitch = item
        strides = []
        for d in range(len(a.shape) - 1, -1, -1):
            strides.append(pitch)
            pitch *= a.shape[d]
            if d == len(a.shape) - 1 and d > 0:
                pitch = (pitch + 15) // 16 * 16
        self.__cuda_array_interface__ = {"shape": tuple(a.shape), "typestr": a.dtype.str, "version": 3,
                                         "data": (a.device_ptr(), False), "strides": tuple(reversed(strides))}


def _view(a):
    return torch.as_tensor(_Memory(a), device="cuda")


class _State:
    """What the program keeps between passes: its context, stores, the graph
    of its steady loop and tensors over the results."""

    def __init__(self, rt):
        self.rt, self.graph, self.step, self.outs, self.keep = rt, None, None, None, []

    def capture(self, body):
        """Issues the loop once (compiling its windows), then records it."""
        body()
        self.rt.capture_begin()
        body()
        self.graph = self.rt.capture_end()

    def __del__(self):
        if self.graph is not None:
            self.rt.graph_destroy(self.graph)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, n, lo, hi, dtype=torch.float64):
    return (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo).to(dtype)


def _poisson(shape):
    """CSR of the 5- or 7-point Laplacian (Dirichlet, row-major, columns ascending)."""
    n, nd = math.prod(shape), len(shape)
    idx = torch.arange(n, device="cuda")
    strides = [math.prod(shape[d + 1:]) for d in range(nd)]
    cols, vals = [], []
    offs = [(d, -1) for d in range(nd)] + [(-1, 0)] + [(d, 1) for d in reversed(range(nd))]
    for d, s in offs:
        if d < 0:
            cols.append(idx)
            vals.append(2.0 * nd)
            continue
        c = idx // strides[d] % shape[d] + s
        cols.append(torch.where((c >= 0) & (c < shape[d]), idx + s * strides[d], -1))
        vals.append(-1.0)
    C = torch.stack(cols, 1)
    mask = C >= 0
    V = torch.tensor(vals, device="cuda", dtype=torch.float64).expand(n, len(vals))
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = mask.sum(1).cumsum(0)
    return rowptr.int(), C[mask].int(), V[mask].contiguous()


def _spd(n, g):
    """CSR of a random symmetric, strictly diagonally dominant matrix: 2 to 13
    off-diagonals drawn per row, symmetrised."""
    k = torch.randint(2, 14, (n,), generator=g, device="cuda").clamp(max=max(0, n - 1))
    r = torch.repeat_interleave(torch.arange(n, device="cuda"), k)
    c = (r + 1 + torch.randint(0, max(1, n - 1), r.shape, generator=g, device="cuda")) % n
    # multiples of 2^-20: every sum below is exact, so no order of addition matters
    v = torch.randint(-(1 << 20), 0, r.shape, generator=g, device="cuda").double() / (1 << 20)
    key, inv = torch.unique(torch.cat([r * n + c, c * n + r]), return_inverse=True)
    vals = torch.zeros(len(key), dtype=torch.float64, device="cuda").index_add_(0, inv, torch.cat([v, v]))
    sums = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, key // n, vals.abs())
    diag = torch.arange(n, device="cuda")
    key = torch.cat([key, diag * n + diag])
    vals = torch.cat([vals, sums + 1.0])
    order = torch.argsort(key)
    key, vals = key[order], vals[order]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return rowptr.int(), (key % n).int(), vals


def _sizes(case):
    """(kind, size) of every problem of a batch: Poisson grids of side 32 to
    mmax or random SPD systems of 1024 to nmax rows, log-uniform."""
    r = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        p, u = r.random(), r.random()
        lo, hi = (32, case["mmax"]) if p < 0.5 else (1024, case["nmax"])
        out.append(("poisson" if p < 0.5 else "spd", int(round(lo * (hi / lo) ** u))))
    return out


def _mult(mat, x):
    """A x in x's precision with torch alone."""
    rp, col, val = mat
    return torch.sparse_csr_tensor(rp.long(), col.long(), val.to(x.dtype), (len(rp) - 1, len(x))) @ x


def _systems(case, seed):
    """Matrices and right-hand sides (b ~ U[-1, 1]) of a solver case, in the
    case's precision."""
    g = _generator(seed)
    if case["kind"] == "cg":
        mats = [_poisson((case["m"],) * 2)]
    elif case["kind"] == "bicg":
        mats = [_poisson((int(m),) * 3) for m in case["sides"].split(",")]
    else:
        mats = [_poisson((s, s)) if k == "poisson" else _spd(s, g) for k, s in _sizes(case)]
    dt = _TORCH[case.get("dtype", "f64")]
    return [((rp, col, val.to(dt)), _uniform(g, len(rp) - 1, -1.0, 1.0, dt)) for rp, col, val in mats]


def _csr(rt, mat):
    return A.CSR(rt, *(t.cpu().numpy() for t in mat))


def _grid(case, seed):
    shape = (case["rows"], case["cols"]) if case["kind"] == "jacobi2d" else (case["m"],) * 3
    g = torch.ones(tuple(s + 2 for s in shape), dtype=_TORCH[case["dtype"]], device="cuda")
    inner = _uniform(_generator(seed), math.prod(shape), 0.0, 1.0, g.dtype).reshape(shape)
    g[tuple(slice(1, -1) for _ in shape)] = inner
    return g


# --------------------------------------------------------------------- cases
def _prepare_bs(case, seed):
    st = _State(_runtime(case["launch"]))
    g, n, rt = _generator(seed), case["n"], st.rt
    data = [_uniform(g, n, lo, hi, torch.float32) for lo, hi in ((5.0, 30.0), (1.0, 100.0), (0.25, 10.0))]
    call, put = torch.empty_like(data[0]), torch.empty_like(data[0])
    torch.cuda.synchronize()
    S, K, T = (rt.wrap(d) for d in data)
    out = (rt.wrap(call), rt.wrap(put))

    def price():
        W.black_scholes(S, K, T, _RATE, _SIGMA, out=out)
        rt.flush()
    if case["graph"]:
        st.capture(price)
    st.step, st.outs, st.keep = price, {"call": call, "put": put}, [S, K, T, out]
    return st


def _prepare_norm(case, seed):
    st = _State(_runtime("default"))
    g, n, rt, dt = _generator(seed), case["n"], st.rt, _TORCH[case["dtype"]]
    x, y = _uniform(g, n, -1.0, 1.0, dt), _uniform(g, n, 0.0, 1.0, dt)
    z, scal = torch.empty_like(x), torch.zeros(3, dtype=dt, device="cuda")
    torch.cuda.synchronize()
    X, Y, Z = rt.wrap(x), rt.wrap(y), rt.wrap(z)
    out = [rt.wrap(scal[i].reshape(())) for i in range(3)]

    def step():
        d = X - Y
        nd = A.norm(d)
        out[0][...] = nd
        out[1][...] = A.asum(Y)
        out[2][...] = A.dot(X, Y)
        Z[...] = d / nd
        del d, nd
        rt.flush()
    st.step, st.outs, st.keep = step, {"z": z, "scalars": scal}, [X, Y, Z, out]
    return st


def _prepare_cg(case, seed):
    st = _State(_runtime(case["launch"]))
    rt = st.rt
    (mat, b), = _systems(case, seed)
    torch.cuda.synchronize()
    Am, B = _csr(rt, mat), rt.wrap(b)
    s = W.cg_start_inplace(B)

    def solve():
        W.cg_reset_inplace(s, B)
        rt.flush()
        for k in range(case["iters"]):
            W.cg_iteration_inplace(Am, s)
            if (k + 1) % case["per_flush"] == 0:
                rt.flush()
        rt.flush()
    st.capture(solve)
    st.outs, st.keep = {"x": _view(s.x), "r": _view(s.r), "rho": _view(s.rho)}, [Am, B, s]
    return st


def _segments(sizes, dtype):
    """One buffer holding a vector per problem, each on a 16-byte boundary."""
    at, total = [], 0
    for n in sizes:
        at.append(total)
        total += (n + 3) // 4 * 4
    flat = torch.zeros(total, dtype=dtype, device="cuda")
    return flat, [flat[o:o + n] for o, n in zip(at, sizes)]


def _prepare_batched(case, seed):
    st = _State(_runtime("batched"))
    rt = st.rt
    systems = _systems(case, seed)
    sizes, dt = [len(b) for _, b in systems], _TORCH[case["dtype"]]
    (x, xs), (r, rs) = _segments(sizes, dt), _segments(sizes, dt)
    torch.cuda.synchronize()
    probs = []
    for (mat, b), xi, ri in zip(systems, xs, rs):
        B = rt.wrap(b)
        s0 = W.cg_start_inplace(B)
        probs.append((_csr(rt, mat), W.CGInPlace(rt.wrap(xi), rt.wrap(ri), s0.p, s0.q, s0.rho), B))
    rt.flush()
    pairs = [(Am, s) for Am, s, _ in probs]

    def solve():
        rt.batch_begin()
        for _, s, B in probs:
            W.cg_reset_inplace(s, B)
            rt.batch_next()
        rt.batch_end()
        for _ in range(case["iters"]):
            W.batched_cg_iteration(rt, pairs)
    st.capture(solve)
    st.outs, st.keep = {"x": x, "r": r}, probs
    return st


def _prepare_bicg(case, seed):
    st = _State(_runtime("serve"))
    rt = st.rt
    systems = _systems(case, seed)
    (x, xs), (r, rs) = (_segments([len(b) for _, b in systems], torch.float64) for _ in range(2))
    torch.cuda.synchronize()
    probs = []
    for (mat, b), xi, ri in zip(systems, xs, rs):
        B = rt.wrap(b)
        s = W.bicgstab_start_inplace(B)
        s.x, s.r = rt.wrap(xi), rt.wrap(ri)
        probs.append((_csr(rt, mat), s, B))
    rt.flush()

    def reset(s, B):
        for a in (s.x, s.p, s.v):
            a[...] = 0.0
        for a in (s.r, s.rhat):
            a[...] = B
        for a in (s.rho, s.alpha, s.omega):
            a[...] = 1.0

    def tick():
        rt.batch_begin()
        for _, s, B in probs:
            reset(s, B)
            rt.batch_next()
        rt.batch_end()
        for _ in range(case["iters"]):
            rt.batch_begin()
            for Am, s, _ in probs:
                W.bicgstab_iteration_inplace(Am, s)
                rt.batch_next()
            rt.batch_end()
    st.capture(tick)
    st.outs, st.keep = {"x": x, "r": r}, probs
    return st


def _prepare_jacobi(case, seed):
    st = _State(_runtime(case["launch"]))
    rt = st.rt
    g = _grid(case, seed)
    torch.cuda.synchronize()
    grid = rt.empty(g.shape, _NUMPY[case["dtype"]])
    two = case["kind"] == "jacobi2d"
    views = W.jacobi_views(grid) if two else W.jacobi3d_views(grid)
    sweep = W.jacobi_sweep if two else W.jacobi3d_sweep

    def sweeps():
        for k in range(case["sweeps"]):
            sweep(views)
            if (k + 1) % case["per_flush"] == 0:
                rt.flush()
        rt.flush()
    start = rt.wrap(g)
    grid[...] = start
    st.capture(sweeps)
    grid[...] = start          # the issued sweeps moved it on
    rt.sync()
    st.outs, st.keep = {"grid": _view(grid)}, [grid, views]
    return st


_PREPARE = {"bs": _prepare_bs, "norm": _prepare_norm, "cg": _prepare_cg, "batched": _prepare_batched,
            "bicg": _prepare_bicg, "jacobi2d": _prepare_jacobi, "jacobi3d": _prepare_jacobi}


def prepare(case, seed):
    st = _PREPARE[case["kind"]](case, seed)
    st.rt.sync()
    return st


def run(state):
    if state.graph is not None:
        state.rt.graph_launch(state.graph)
    else:
        state.step()
    return state.outs


def _rows_nnz(case):
    if case["kind"] == "cg":
        m = case["m"]
        return [(m * m, 5 * m * m - 4 * m)]
    if case["kind"] == "bicg":
        return [(m ** 3, 7 * m ** 3 - 6 * m * m) for m in map(int, case["sides"].split(","))]
    # a random SPD row holds about 15 merged off-diagonals and its diagonal
    return [(s * s, 5 * s * s - 4 * s) if k == "poisson" else (s, 16 * s) for k, s in _sizes(case)]


def work(case):
    kind = case["kind"]
    if kind == "bs":
        return {"bytes": 20 * case["n"], "flops": 60 * case["n"]}
    e = 4 if case.get("dtype", "f64") == "f32" else 8
    if kind == "norm":
        return {"bytes": 3 * e * case["n"], "flops": 7 * case["n"]}
    if kind in ("jacobi2d", "jacobi3d"):
        two = kind == "jacobi2d"
        cells = case["rows"] * case["cols"] if two else case["m"] ** 3
        return {"bytes": 2 * e * cells * case["sweeps"], "flops": (5 if two else 7) * cells * case["sweeps"]}
    rows = sum(n for n, _ in _rows_nnz(case))
    nnz = sum(z for _, z in _rows_nnz(case))
    matrix = (4 + e) * nnz + 4 * rows
    if kind == "bicg":
        # two products; the vector passes of the six dependent phases
        return {"bytes": case["iters"] * (2 * matrix + 20 * e * rows), "flops": case["iters"] * (4 * nnz + 24 * rows)}
    return {"bytes": case["iters"] * (matrix + 10 * e * rows), "flops": case["iters"] * (2 * nnz + 10 * rows)}


# --------------------------------------------------------------------- exact
def _exact_cg(mat, b, iters):
    b = b.double()
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rho = r @ r
    for _ in range(iters):
        q = _mult(mat, p)
        alpha = rho / (p @ q)
        x = x + alpha * p
        r = r - alpha * q
        new = r @ r
        p = r + new / rho * p
        rho = new
    return x, r, rho


def _exact_bicg(mat, b, iters):
    x, r, rhat, p, v = torch.zeros_like(b), b.clone(), b.clone(), torch.zeros_like(b), torch.zeros_like(b)
    rho = alpha = omega = torch.ones((), dtype=b.dtype, device="cuda")
    for _ in range(iters):
        new = rhat @ r
        p = r + new / rho * (alpha / omega) * (p - omega * v)
        v = _mult(mat, p)
        alpha = new / (rhat @ v)
        s = r - alpha * v
        t = _mult(mat, s)
        omega = (t @ s) / (t @ t)
        x = x + alpha * p + omega * s
        r = s - omega * t
        rho = new
    return x, r


def exact(case, seed):
    kind = case["kind"]
    if kind == "bs":
        g, n = _generator(seed), case["n"]
        S, K, T = (_uniform(g, n, lo, hi, torch.float32).double()
                   for lo, hi in ((5.0, 30.0), (1.0, 100.0), (0.25, 10.0)))
        v = _SIGMA * T.sqrt()
        d1 = ((S / K).log() + (_RATE + 0.5 * _SIGMA * _SIGMA) * T) / v
        d2 = d1 - v
        kd = K * torch.exp(-_RATE * T)

        def cdf(d):
            return 0.5 * torch.special.erfc(d * -math.sqrt(0.5))
        return {"call": S * cdf(d1) - kd * cdf(d2), "put": kd * cdf(-d2) - S * cdf(-d1)}
    if kind == "norm":
        g, n, dt = _generator(seed), case["n"], _TORCH[case["dtype"]]
        x, y = _uniform(g, n, -1.0, 1.0, dt).double(), _uniform(g, n, 0.0, 1.0, dt).double()
        d = x - y
        nd = d.square().sum().sqrt()
        return {"z": d / nd, "scalars": torch.stack([nd, y.sum(), x @ y])}
    if kind in ("jacobi2d", "jacobi3d"):
        g = _grid(case, seed).double()
        nd = g.dim()
        mid = tuple(slice(1, -1) for _ in range(nd))
        for _ in range(case["sweeps"]):
            acc = g[mid].clone()
            for d in range(nd):
                for lo, hi in ((0, -2), (2, None)):
                    acc += g[mid[:d] + (slice(lo, hi),) + mid[d + 1:]]
            g[mid] = acc / (2 * nd + 1)
        return {"grid": g}
    systems = _systems(case, seed)
    if kind == "cg":
        x, r, rho = _exact_cg(systems[0][0], systems[0][1], case["iters"])
        return {"x": x, "r": r, "rho": rho}
    (x, xs), (r, rs) = (_segments([len(b) for _, b in systems], torch.float64) for _ in range(2))
    for (mat, b), xi, ri in zip(systems, xs, rs):
        sol = _exact_bicg(mat, b, case["iters"]) if kind == "bicg" else _exact_cg(mat, b, case["iters"])
        xi.copy_(sol[0])
        ri.copy_(sol[1])
    return {"x": x, "r": r}
