"""The work that users of this framework have it do, as cases that can be timed.

A case is one call (or one burst of calls) through the public entry points of
``paper_2606_07004_gb300.binding``: log-determinant solves over the methods,
precisions, operators and sizes that the estimators are used with, a graph
plan's replay, a burst through the continuous-batching server, and the sketch
orthogonalisation.  ``listed`` names them; ``draw`` gives others of the same
ranges.  Matrices are generated on the GPU from the seed (it moves the
diagonal and draws the probes) and handed over as a user's program would:
host CSR arrays, or device arrays for the graphs.

A mixed-precision solve's estimates carry FP32 rounding, so they are returned
as FP32 numbers; FP64 solves return FP64.  The double-float mode returns FP32
as well: its matrix values are FP32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_07004_gb300 import binding as B
from paper_2606_07004_gb300 import grf

PRECISION = {"fp64": B.FP64, "fp32": B.MIXED_FP32, "f32x2": B.MIXED_F32X2}


def listed():
    return [
        # One estimate on a small grid, a fresh call each time: launches and
        # dependent round trips set the time.
        dict(name="small_lap2d_fp64", kind="solve", matrix="lap2d", nx=64, ny=64, nz=1,
             method="oslq", window=0, precision="fp64", probes=30, steps=30),
        # A hyper-parameter loop that replays one captured solve with new
        # seeds (odd, ragged grid; the paper's OSA-IOP setting).
        dict(name="plan_lap2d_fp32", kind="plan", matrix="lap2d", nx=211, ny=150, nz=1,
             method="osaiop", window=2, precision="fp32", probes=21, steps=20),
        # The FP64 estimators on a 2M-row 3D Laplacian: OSLQ ...
        dict(name="lap3d_128_fp64_oslq", kind="solve", matrix="lap3d", nx=128, ny=128, nz=128,
             method="oslq", window=0, precision="fp64", probes=60, steps=50),
        # ... and OSA-IOP with a window of four vectors.
        dict(name="lap3d_128_fp64_iop4", kind="solve", matrix="lap3d", nx=128, ny=128, nz=128,
             method="osaiop", window=4, precision="fp64", probes=60, steps=50),
        # The SPDE Matern precision in mixed FP32, many probes.
        dict(name="matern_1024_fp32", kind="solve", matrix="matern", nx=1024, ny=1024, nz=1,
             method="oslq", window=0, precision="fp32", probes=120, steps=80),
        # The largest serving request alone: 4M rows, narrow blocks, odd side.
        dict(name="lap3d_159_fp32", kind="solve", matrix="lap3d", nx=159, ny=159, nz=159,
             method="oslq", window=0, precision="fp32", probes=30, steps=50),
        # Several diagonal shifts of one power-law graph Laplacian.
        dict(name="graph_1m_shifts_fp32", kind="shifts", matrix="graph", nx=1000003, ny=1, nz=1,
             method="osaiop", window=4, precision="fp32", probes=64, steps=40, shifts=4),
        # The same kind of graph within the error budget: double-float vectors.
        dict(name="graph_300k_f32x2", kind="solve", matrix="graph", nx=300007, ny=1, nz=1,
             method="osaiop", window=4, precision="f32x2", probes=64, steps=60),
        # One candidate of the Gaussian-random-field likelihood on the paper's
        # grid: log-determinant (its OSA-IOP setting) and quadratic form.
        dict(name="grf_900x1200_fp32", kind="grf", matrix="wendland", nx=1200, ny=900, nz=1,
             theta=50.0, method="osaiop", window=2, precision="fp32", probes=21, steps=20),
        # The FP64 check of such a candidate on a smaller, odd grid.
        dict(name="grf_240x301_fp64", kind="grf", matrix="wendland", nx=301, ny=240, nz=1,
             theta=20.0, method="oslq", window=0, precision="fp64", probes=30, steps=30),
        # A burst of requests of mixed sizes through the server.
        dict(name="serve_burst_fp32", kind="serve", requests=12, n_lo=10000, n_hi=1000000, mix=3,
             precision="fp32", probes=30, steps=50),
        # The Hutch++ orthogonalisation step by itself.
        dict(name="orth_1m_fp64", kind="orth", n=1000003, s=20, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "plan", "shifts", "grf", "serve", "orth"])
    if kind == "orth":
        return dict(kind="orth", n=_log_int(rng, 5000, 2000000), s=rng.randint(5, 40),
                    precision=rng.choice(["fp64", "fp32"]))
    if kind == "serve":
        return dict(kind="serve", requests=rng.randint(4, 12), n_lo=10000,
                    n_hi=_log_int(rng, 50000, 1000000), mix=rng.randrange(1000), precision="fp32",
                    probes=rng.choice([21, 30, 45]), steps=rng.randint(20, 50))
    method = rng.choice(["oslq", "osaiop"])
    c = dict(kind=kind, method=method, window=rng.choice([2, 4, 8]) if method == "osaiop" else 0)
    if kind == "grf":
        ny = _log_int(rng, 100, 900)
        return dict(c, matrix="wendland", nx=ny + rng.randint(0, 300), ny=ny, nz=1,
                    theta=round(rng.uniform(10.0, 20.0 if ny < 300 else 50.0), 1),
                    precision="fp64" if ny < 240 else "fp32", probes=rng.choice([21, 30]),
                    steps=rng.randint(12, 20 if ny > 400 else 30))
    if kind == "shifts":
        return dict(c, matrix="graph", nx=_log_int(rng, 30000, 600000), ny=1, nz=1,
                    precision=rng.choice(["fp32", "f32x2"]), probes=rng.choice([21, 30, 64]),
                    steps=rng.randint(15, 40), shifts=rng.randint(2, 4))
    c["precision"] = rng.choice(["fp64", "fp32", "fp32"])
    c["probes"] = rng.choice([21, 30, 45, 60])
    c["steps"] = rng.randint(15, 50)
    top = 40000 if kind == "plan" else 2000000
    shape = rng.choice(["lap2d", "lap3d", "matern"] + (["graph"] if kind == "solve" else []))
    n = _log_int(rng, 4000, top)
    if shape == "lap3d":
        s = max(9, round(n ** (1 / 3)))
        return dict(c, matrix=shape, nx=s + rng.randint(0, 4), ny=s, nz=max(5, s - rng.randint(0, 4)))
    if shape == "lap2d":
        s = round(math.sqrt(n))
        return dict(c, matrix=shape, nx=s + rng.randint(0, 30), ny=s, nz=1)
    if shape == "matern":
        s = round(math.sqrt(n))
        return dict(c, matrix=shape, nx=s, ny=s, nz=1)
    return dict(c, matrix="graph", nx=min(max(n, 30000), 600000), ny=1, nz=1,
                precision=rng.choice(["fp64", "f32x2"]))


# ---- matrices ---------------------------------------------------------------

def _stencil(c, seed):
    """CSR on the GPU of a Dirichlet grid stencil (x fastest), diagonal moved
    by the seed: (n, rowptr, colind, vals)."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    n = nx * ny * nz
    u = 1.0 + (seed % 1009) / 1009.0
    i = torch.arange(n, device="cuda")
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    if c["matrix"] == "matern":
        k = 4.0 + 0.05 * u
        near = (y > 0).double() + (x > 0).double() + (x < nx - 1).double() + (y < ny - 1).double()
        taps = [(0, -2, 0, 1.0), (-1, -1, 0, 2.0), (0, -1, 0, -2 * k), (1, -1, 0, 2.0),
                (-2, 0, 0, 1.0), (-1, 0, 0, -2 * k), (0, 0, 0, k * k + near), (1, 0, 0, -2 * k),
                (2, 0, 0, 1.0), (-1, 1, 0, 2.0), (0, 1, 0, -2 * k), (1, 1, 0, 2.0), (0, 2, 0, 1.0)]
    elif c["matrix"] == "lap3d":
        taps = [(0, 0, -1, -1.0), (0, -1, 0, -1.0), (-1, 0, 0, -1.0), (0, 0, 0, 6.0 + 0.01 * u),
                (1, 0, 0, -1.0), (0, 1, 0, -1.0), (0, 0, 1, -1.0)]
    else:
        taps = [(0, -1, 0, -1.0), (-1, 0, 0, -1.0), (0, 0, 0, 4.0 + 0.1 * u), (1, 0, 0, -1.0),
                (0, 1, 0, -1.0)]
    ok = torch.empty(n, len(taps), dtype=torch.bool, device="cuda")
    col = torch.empty(n, len(taps), dtype=torch.int32, device="cuda")
    val = torch.empty(n, len(taps), dtype=torch.float64, device="cuda")
    for t, (dx, dy, dz, v) in enumerate(taps):
        ok[:, t] = ((x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny)
                    & (z + dz >= 0) & (z + dz < nz))
        col[:, t] = i + (dx + nx * (dy + ny * dz))
        val[:, t] = v
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ok.sum(1), 0, out=ptr[1:])
    return n, ptr.int(), col[ok], val[ok]


def _graph(c, seed):
    """CSR on the GPU of a Chung-Lu power-law graph Laplacian (exponent 2.3,
    mean degree 8, hubs first); with kind "solve" plus a small diagonal."""
    n, mean = c["nx"], 8.0
    g = 1.0 / 1.3
    lo, hi = 1e-9, float(n)
    for _ in range(200):  # the offset at which the largest expected degree is sqrt(n mean)
        mid = 0.5 * (lo + hi)
        avg = ((n + mid) ** (1 - g) - mid ** (1 - g)) / ((1 - g) * n)
        lo, hi = (mid, hi) if mid ** (-g) / avg > math.sqrt(n * mean) / mean else (lo, mid)
    w = (torch.arange(n, device="cuda", dtype=torch.float64) + hi) ** (-g)
    cdf = torch.cumsum(w / w.sum(), 0)
    r = torch.Generator(device="cuda").manual_seed(seed)
    e = torch.rand(2, int(n * mean / 2), generator=r, device="cuda", dtype=torch.float64)
    u, v = torch.searchsorted(cdf, e).clamp_(max=n - 1)
    u, v = u[u != v], v[u != v]
    i = torch.arange(n, device="cuda")
    key = torch.unique(torch.cat([u * n + v, v * n + u, i * (n + 1)]))
    row, col = key // n, key % n
    cnt = torch.bincount(row, minlength=n)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(cnt, 0, out=ptr[1:])
    shift = 0.0 if c["kind"] == "shifts" else 0.02
    val = torch.where(row == col, (cnt - 1).double()[row] + shift, -1.0)
    return n, ptr.int(), col.int(), val


def _csr(c, seed):
    return _graph(c, seed) if c["matrix"] == "graph" else _stencil(c, seed)


def _handle(c, seed):
    if c["matrix"] == "wendland":
        return B.Handle.grid(c["nx"], c["ny"], _table(c, seed))
    n, ptr, col, val = _csr(c, seed)
    if c["matrix"] == "graph":
        torch.cuda.synchronize()
        return B.Handle(n, ptr, col, val, device=True)
    return B.Handle(n, ptr.cpu().numpy(), col.cpu().numpy(), val.cpu().numpy())


def _table(c, seed):
    return grf.wendland_table(c["theta"], 0.1 * (1.0 + (seed % 1009) / 1009.0))


def _field(c, seed):
    r = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(c["nx"] * c["ny"], generator=r, device="cuda", dtype=torch.float64)


def _shifts(c, seed):
    r = np.random.default_rng(seed)
    return r.uniform(1e-3, 1e-1, c["shifts"])


def _requests(c):
    """The server's requests: kinds and log-uniform sizes, the same for every seed."""
    r = np.random.default_rng(c["mix"])
    out = []
    for k in range(c["requests"]):
        n = math.exp(r.uniform(math.log(c["n_lo"]), math.log(c["n_hi"])))
        m = ["lap2d", "lap3d", "matern"][int(r.integers(3))]
        s = max(6, round(n ** (1 / 3))) if m == "lap3d" else max(6, round(math.sqrt(n)))
        out.append(dict(kind="solve", matrix=m, nx=s, ny=s, nz=s if m == "lap3d" else 1,
                        method="oslq", window=0, precision=c["precision"], probes=c["probes"],
                        steps=c["steps"]))
    return out


def _block(c, seed):
    """A sketch-like block: random signs smoothed along the rows."""
    r = torch.Generator(device="cuda").manual_seed(seed)
    y = torch.randint(0, 2, (c["n"] + 2, c["s"]), generator=r, device="cuda").double() * 2 - 1
    y = y[1:-1] * 0.6 - y[:-2] * 0.2 - y[2:] * 0.2
    return y.contiguous() if c["precision"] == "fp64" else y.float().contiguous()


# ---- the calls --------------------------------------------------------------

def prepare(case, seed):
    c = case
    if c["kind"] == "orth":
        y = _block(c, seed)
        return dict(case=c, y=y, a=torch.empty_like(y))
    if c["kind"] == "serve":
        reqs = _requests(c)
        return dict(case=c, seed=seed, reqs=reqs, server=B.Server(32 << 30),
                    handles=[_handle(q, seed + i) for i, q in enumerate(reqs)])
    s = dict(case=c, seed=seed, handle=_handle(c, seed))
    if c["kind"] == "plan":
        s["plan"] = B.Plan(s["handle"], B.METHOD_OSAIOP if c["method"] == "osaiop" else B.METHOD_OSLQ,
                           c["probes"], c["steps"], c["window"], precision=PRECISION[c["precision"]])
    if c["kind"] == "shifts":
        s["shifts"] = _shifts(c, seed)
    if c["kind"] == "grf":
        s["field"] = _field(c, seed)
    return s


def _numbers(results, precision):
    """Estimates, their two terms and the quadratic forms of the probes."""
    t = np.float64 if precision == "fp64" else np.float32
    return dict(logdet=np.array([r.logdet for r in results], t),
                tr_sub=np.array([r.tr_sub for r in results], t),
                tr_res=np.array([r.tr_res for r in results], t),
                forms=np.concatenate([r.per_probe for r in results]).astype(t),
                norms=np.concatenate([r.z_norm2 for r in results]).astype(t),
                rank=np.array([r.s_eff for r in results], np.int32))


def run(state):
    c = state["case"]
    if c["kind"] == "orth":
        f = B.logdet_orth if c["precision"] == "fp64" else B.logdet_orth_f32
        rank = f(c["n"], c["s"], state["y"], c["s"], state["a"], c["s"])
        return dict(a=state["a"], rank=rank)
    p = PRECISION[c["precision"]]
    if c["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(h, B.METHOD_OSLQ, q["probes"], q["steps"], seed=state["seed"] + i,
                          precision=p)
               for i, (h, q) in enumerate(zip(state["handles"], state["reqs"]))]
        out = [srv.wait(i) for i in ids]
        for i in ids:
            srv.release(i)
        return _numbers(out, c["precision"])
    h = state["handle"]
    if c["kind"] == "plan":
        return _numbers([state["plan"].run(state["seed"])], c["precision"])
    if c["kind"] == "shifts":
        f = h.osaiop_shifts if c["method"] == "osaiop" else h.oslq_shifts
        return _numbers(f(state["shifts"], c["probes"], c["steps"], iop_window=c["window"],
                          seed0=state["seed"], precision=p), c["precision"])
    f = h.osaiop if c["method"] == "osaiop" else h.oslq
    out = _numbers([f(c["probes"], c["steps"], iop_window=c["window"], seed=state["seed"],
                      precision=p)], c["precision"])
    if c["kind"] == "grf":
        out["quad"] = h.quadform(state["field"])
    return out


# ---- what a pass cannot do without ------------------------------------------

def _nnz(c):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["matrix"] == "graph":
        return 9 * nx
    if c["matrix"] == "wendland":
        return 0
    return {"lap2d": 5, "lap3d": 7, "matern": 13}[c["matrix"]] * nx * ny * nz


def work(case):
    """Per Krylov step the matrix read once, the newest and the other window
    vectors read once, the new vector written once; the multiply-adds of the
    product, the dots and the window.  A gridded operator has no stored matrix
    and is counted as a fast convolution."""
    c = case
    if c["kind"] == "orth":
        e = 8 if c["precision"] == "fp64" else 4
        return {"bytes": 2.0 * e * c["n"] * c["s"], "flops": 2.0 * c["n"] * c["s"] ** 2}
    if c["kind"] == "serve":
        w = [work(q) for q in _requests(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    e = {"fp64": 8, "fp32": 4, "f32x2": 8}[c["precision"]]
    n = c["nx"] * c["ny"] * c["nz"]
    s = c["probes"] // 3
    r = c["probes"] - 2 * s
    members = c.get("shifts", 1)
    cols = members * (s + r + (s if c["method"] == "osaiop" else 0))
    phases = 2 if c["method"] == "osaiop" else 1
    k = c["window"] or 2
    nnz = _nnz(c)
    value = 8 if c["precision"] == "fp64" else 4
    product = 2.0 * nnz if nnz else 10.0 * n * math.log2(n)
    return {"bytes": c["steps"] * (phases * nnz * (value + 4.0) + n * cols * e * (k + 1.0)),
            "flops": c["steps"] * cols * (product + 2.0 * n * (2 * k + 1))}


# ---- 64-bit values ----------------------------------------------------------

_M64 = (1 << 64) - 1


def _signed(v):
    v &= _M64
    return v - (1 << 64) if v >> 63 else v


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _mix(z):
    """SplitMix64's output function on int64 tensors (wrapping)."""
    z = (z ^ _shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _signs(seed, stream, n, b):
    gold = _signed(0x9E3779B97F4A7C15)
    key = _mix(torch.tensor([_signed(seed + (stream + 1) * 0x9E3779B97F4A7C15)], device="cuda"))
    row = torch.arange(1, n + 1, device="cuda")[:, None]
    col = torch.arange(b, device="cuda")[None, :] << 32
    return 1.0 - 2.0 * (_mix(key + (row + col) * gold) < 0).double()


def _qr(y):
    q, r = torch.linalg.qr(y)
    return q * torch.sign(torch.diagonal(r))


def _dot(a, b):
    return (a * b).sum(0)


def _lanczos_forms(apply, v, m):
    """sum tau^2 log(theta) of m Lanczos steps for each (normalised) column."""
    al, be = [], []
    v = v / v.norm(dim=0)
    prev, beta = None, None
    for j in range(m):
        w = apply(v)
        a = _dot(v, w)
        w = w - a * v - (beta * prev if prev is not None else 0.0)
        al.append(a)
        if j + 1 < m:
            beta = w.norm(dim=0)
            be.append(beta)
            prev, v = v, w / beta
    al = torch.stack(al, 1).cpu().numpy()
    be = torch.stack(be, 1).cpu().numpy() if be else np.zeros((al.shape[0], 0))
    out = []
    for a, b in zip(al, be):
        th, u = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
        out.append(float((u[0] ** 2 * np.log(th)).sum()))
    return np.array(out)


def _iop(apply, v, m, k):
    """m steps of Arnoldi with a window of k vectors: the basis (unless only
    its first column's products are wanted) and log(H) e_1 per column."""
    b = v.shape[1]
    beta = v.norm(dim=0)
    V = [v / beta]
    H = np.zeros((b, m + 1, m))
    for j in range(m):
        w = apply(V[j])
        for i in range(max(0, j - k + 1), j + 1):
            h = _dot(V[i], w)
            w = w - h * V[i]
            H[:, i, j] = h.cpu().numpy()
        h = w.norm(dim=0)
        H[:, j + 1, j] = h.cpu().numpy()
        if j + 1 < m:
            V.append(w / h)
    c = np.zeros((b, m))
    for p in range(b):
        th, U = np.linalg.eig(H[p, :m, :])
        e1 = np.zeros(m)
        e1[0] = 1.0
        c[p] = np.real(U @ (np.log(th.astype(complex)) * np.linalg.solve(U, e1)))
    return V, beta, torch.tensor(c, device="cuda")


def _operator(c, seed, shift=0.0):
    """(n, X -> Q X in FP64, Gershgorin interval) by plain torch."""
    if c["matrix"] == "wendland":
        nx, ny, t = c["nx"], c["ny"], torch.tensor(_table(c, seed), device="cuda")
        R = t.shape[0] - 1
        my, mx = ny + R, nx + R
        w = torch.zeros(my, mx, dtype=torch.float64, device="cuda")
        d = torch.arange(-R, R + 1, device="cuda")
        py, px = d[abs(d) < ny], d[abs(d) < nx]
        w[(py % my)[:, None], (px % mx)[None, :]] = t[py.abs()][:, px.abs()]
        f = torch.fft.rfft2(w)
        yc, xc = ny // 2, nx // 2
        inner = t[d[(yc + d >= 0) & (yc + d < ny)].abs()][:, d[(xc + d >= 0) & (xc + d < nx)].abs()]
        rad = float(inner.abs().sum() - t[0, 0].abs())

        def apply(X):
            out = torch.empty_like(X)
            for p in range(X.shape[1]):
                z = torch.fft.rfft2(X[:, p].reshape(ny, nx), s=(my, mx))
                out[:, p] = torch.fft.irfft2(z * f, s=(my, mx))[:ny, :nx].reshape(-1)
            return out
        return nx * ny, apply, float(t[0, 0]) - rad, float(t[0, 0]) + rad
    n, ptr, col, val = _csr(c, seed)
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), torch.diff(ptr.long()))
    diag = row == col
    val = val + shift * diag
    d = val[diag]
    rad = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, (val * ~diag).abs())
    A = torch.sparse_csr_tensor(ptr, col, val, size=(n, n))
    return n, (lambda X: A @ X), float((d - rad).min()), float((d + rad).max())


def _estimate(c, seed, matrix_seed, shift=0.0):
    n, q, lo, hi = _operator(c, matrix_seed, shift)
    if lo <= 0:
        lo = 1e-6 * hi
    s = c["probes"] // 3
    r = c["probes"] - 2 * s
    m, k = c["steps"], c["window"]
    S, G = _signs(seed, 0, n, s), _signs(seed, 1, n, r)
    if c["method"] == "oslq":
        scale = hi
        apply = lambda X: q(X) / hi  # noqa: E731
        Y = apply(S)
        A = _qr(Y)
        Z = G - A @ (A.T @ G)
        zn = _dot(Z, Z).cpu().numpy()
        forms = _lanczos_forms(apply, torch.cat([A, Z], 1), m)
    else:
        scale, gamma = lo, math.sqrt(lo * hi)
        more = math.log(gamma / lo)
        apply = lambda X: q(X) / gamma  # noqa: E731
        V, beta, cs = _iop(apply, S, m, k)
        Y = more * S
        for j, v in enumerate(V):
            Y += beta * cs[:, j] * v
        del V
        A = _qr(Y)
        Z = G - A @ (A.T @ G)
        zn = _dot(Z, Z).cpu().numpy()
        X = torch.cat([A, Z], 1)
        V, beta, cs = _iop(apply, X, m, k)
        f = torch.zeros(s + r, dtype=torch.float64, device="cuda")
        for j, v in enumerate(V):
            f += cs[:, j] * _dot(V[0], v)
        forms = f.cpu().numpy() + more
    sub, res = forms[:s].sum(), (zn * forms[s:]).mean()
    return dict(logdet=n * math.log(scale) + sub + res, tr_sub=sub, tr_res=res, forms=forms, norms=zn)


def exact(case, seed):
    c = case
    if c["kind"] == "orth":
        return dict(a=_qr(_block(c, seed).double()), rank=None)
    if c["kind"] == "serve":
        got = [_estimate(q, seed + i, seed + i) for i, q in enumerate(_requests(c))]
    elif c["kind"] == "shifts":
        got = [dict(_estimate(c, seed + t, seed, shift=float(x)), forms=np.zeros(0), norms=np.zeros(0))
               for t, x in enumerate(_shifts(c, seed))]
    else:
        got = [_estimate(c, seed, seed)]
    out = {k: np.array([g[k] for g in got]) for k in ("logdet", "tr_sub", "tr_res")}
    out |= {k: np.concatenate([g[k] for g in got]) for k in ("forms", "norms")}
    out["rank"] = None
    if c["kind"] == "grf":
        x = _field(c, seed)[:, None]
        out["quad"] = float(_dot(x, _operator(c, seed)[1](x))[0])
    return out
