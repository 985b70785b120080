"""Performance cases: the work a user has this library do, through its public calls.

The path is: kNN and row order -> MVGD rows -> products and solves of (I - L) u = f, on one cloud, on a
batch of uneven clouds, on closed and open surfaces, in FP64 and in the FP32 hi + lo format.  Each case
is a stage or a whole pass of it, at the sizes of the test workloads: the Fibonacci sphere of 2,562 points,
the random sphere of 1,048,576, the torus of 524,288, batches of uneven clouds, and sizes between them.

Solves ask for 1e-10, the tolerance of the Fibonacci workload and of the eigensolver's inner solves.
"""
import math

import numpy as np
import torch

from paper_1603_04100_gb300 import api
from paper_1603_04100_gb300.batch import BatchPipeline
from paper_1603_04100_gb300.pipeline import Pipeline

RTOL = 1e-10
SLICE = 32
N_RHS = 8
PREC = {"fp64": api.FP64, "fp32": api.FP32_REFINE}
DENSE_MAX = 20_500      # rows up to which exact() solves the dense system
DENSE_MAX_BATCH = 8_000


def listed():
    return [
        # the smallest use: rows of a small lattice and L applied to the coordinates (exact value -2 x)
        dict(name="rows_small", kind="rows", shape="fibonacci", n=2562, k=12, prec="fp64"),
        # its solve, by plain BiCGSTAB: latency of the smallest system
        dict(name="solve_small", kind="solve", shape="fibonacci", n=2562, k=12, prec="fp64", nrhs=1, precond=0),
        # one request of a serving mix: a small cloud with several right-hand sides, points to solution
        dict(name="cloud_small", kind="cloud", shape="torus", n=7001, k=16, prec="fp32", nrhs=4),
        # an open surface call by call: kNN, rows, Dirichlet rows on the rim, multigrid-preconditioned solve
        dict(name="open_surface", kind="open", shape="hemisphere", n=20_000, k=20, prec="fp32", nrhs=1),
        # a block of the eigensolver's shift-invert step: 8 right-hand sides, the hierarchy kept
        dict(name="block_solve", kind="solve", shape="sphere", n=16_000, k=20, prec="fp64", nrhs=8, precond=2),
        # neighbour search of the largest cloud
        dict(name="knn_large", kind="knn", shape="sphere", n=1_048_576, k=20),
        # rows of the largest cloud, mixed format
        dict(name="rows_large_mixed", kind="assemble", shape="sphere", n=1_048_576, k=20, prec="fp32"),
        # rows of the torus with the widest stencil, FP64
        dict(name="rows_torus_fp64", kind="assemble", shape="torus", n=524_288, k=24, prec="fp64"),
        # the product an FP32 Krylov solve repeats
        dict(name="product_f32", kind="spmv", shape="sphere", n=1_048_576, k=20, prec="fp32", mode="f32", nrhs=1),
        # the FP64 product of several vectors, a ragged size
        dict(name="product_f64", kind="spmv", shape="torus", n=100_003, k=16, prec="fp64", mode="f64", nrhs=4),
        # a batch of uneven clouds with four right-hand sides each
        dict(name="batch", kind="batch", count=32, n_lo=2000, n_hi=65_536, k=20, prec="fp32", nrhs=4, mix=1),
        # the headline: the largest cloud from points to solution
        dict(name="cloud_large", kind="cloud", shape="sphere", n=1_048_576, k=20, prec="fp32", nrhs=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rows", "solve", "solve", "cloud", "cloud", "open", "knn", "assemble", "spmv", "batch"])
    shape = rng.choice(["sphere", "ellipsoid", "torus"])
    k = rng.choice([16, 20, 24])
    prec = rng.choice(["fp64", "fp32"])
    if kind == "rows":
        return dict(kind=kind, shape=shape, n=_log_int(rng, 2000, 60_000), k=k, prec="fp64")
    if kind == "solve":
        precond = rng.choice([0, 1, 2, 2])
        return dict(kind=kind, shape=shape, n=_log_int(rng, 1000, 100_000 if precond == 2 else 20_000), k=k,
                    prec=prec, nrhs=rng.randint(1, 8), precond=precond)
    if kind == "cloud":
        n = _log_int(rng, 1000, 1_000_000)
        return dict(kind=kind, shape=shape, n=n, k=k, prec="fp32", nrhs=1 if n > 200_000 else rng.randint(1, 8))
    if kind == "open":
        return dict(kind=kind, shape="hemisphere", n=_log_int(rng, 3000, 60_000), k=20, prec=prec, nrhs=1)
    if kind == "knn":
        return dict(kind=kind, shape=shape, n=_log_int(rng, 1000, 1_048_576), k=rng.randint(8, 31))
    if kind == "assemble":
        return dict(kind=kind, shape=shape, n=_log_int(rng, 2000, 500_000), k=rng.choice([12, 16, 20, 24, 31]),
                    prec=prec)
    if kind == "spmv":
        mode = "f64" if prec == "fp64" else rng.choice(["f32", "hilo"])
        return dict(kind=kind, shape=shape, n=_log_int(rng, 2000, 1_000_000), k=rng.choice([12, 16, 20, 24, 31]),
                    prec=prec, mode=mode, nrhs=rng.randint(1, 8))
    return dict(kind="batch", count=rng.randint(4, 24), n_lo=2000, n_hi=50_000, k=k, prec="fp32",
                nrhs=rng.randint(1, 4), mix=rng.randint(2, 1 << 20))


# ---------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, *size):
    return torch.rand(*size, dtype=torch.float64, device="cuda", generator=g)


def _sphere(n, g):
    p = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=g)
    return (p / p.norm(dim=1, keepdim=True)).contiguous()


def _points(shape, n, seed):
    """(points, boundary flags or None): the surfaces of the test workloads, drawn from the seed."""
    g = _gen(seed)
    if shape == "sphere":
        return _sphere(n, g), None
    if shape == "ellipsoid":
        return (_sphere(n, g) * torch.tensor([1.0, 0.7, 0.4], dtype=torch.float64, device="cuda")).contiguous(), None
    if shape == "torus":  # R = 1, r = 0.4, parameter density proportional to 1 + 0.75 cos(theta)
        m = int(2.0 * n) + 4096
        th, ph, u = 2 * math.pi * _rand(g, m), 2 * math.pi * _rand(g, m), _rand(g, m)
        keep = 1.75 * u < 1.0 + 0.75 * torch.cos(th)
        th, ph = th[keep][:n], ph[keep][:n]
        rho = 1.0 + 0.4 * torch.cos(th)
        return torch.stack([rho * torch.cos(ph), rho * torch.sin(ph), 0.4 * torch.sin(th)], 1).contiguous(), None
    if shape == "hemisphere":  # a rim of evenly spaced boundary points, random points above it
        nb = int(round(math.sqrt(2.0 * math.pi * n) / 2.0))
        t = (torch.arange(nb, dtype=torch.float64, device="cuda") + _rand(g, 1)) * (2.0 * math.pi / nb)
        p = _sphere(int(2.2 * (n - nb)) + 4096, g)
        p = p[p[:, 2] > 0.0][: n - nb]
        rim = torch.stack([torch.cos(t), torch.sin(t), torch.zeros_like(t)], 1)
        flags = torch.zeros(n, dtype=torch.uint8, device="cuda")
        flags[:nb] = 1
        return torch.cat([rim, p]).contiguous(), flags
    # the Fibonacci lattice in an orientation of the seed's
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    z = 1.0 - (2.0 * i + 1.0) / n
    ph = 2.0 * math.pi * i / ((1.0 + math.sqrt(5.0)) / 2.0)
    rho = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    p = torch.stack([rho * torch.cos(ph), rho * torch.sin(ph), z], 1)
    a = torch.randn(3, 3, dtype=torch.float64, device="cuda", generator=g)
    e0 = a[0] / a[0].norm()
    e1 = a[1] - (a[1] @ e0) * e0
    e1 = e1 / e1.norm()
    return (p @ torch.stack([e0, e1, torch.linalg.cross(e0, e1)])).contiguous(), None


def _rhs(p, q):
    """q smooth right-hand sides, [n][q]."""
    x, y, z = p[:, 0], p[:, 1], p[:, 2]
    cols = [13.0 * (5.0 * z ** 3 - 3.0 * z), x, y * z, x * x - y * y, torch.sin(x) * torch.exp(y), z, x * y, 1.0 + x * z]
    return torch.stack(cols[:q], 1).contiguous()


def _vectors(n, q, seed, dtype):
    """Vectors a Krylov solve multiplies: a smooth part and noise, stored order."""
    g = _gen(seed + 77)
    t = torch.arange(n, dtype=torch.float64, device="cuda")[:, None] / n
    x = torch.sin(6.0 * t + torch.arange(q, dtype=torch.float64, device="cuda")) + 0.1 * torch.randn(
        n, q, dtype=torch.float64, device="cuda", generator=g)
    return x.to(dtype).contiguous()


def _batch_sizes(case):
    rng = np.random.Generator(np.random.PCG64(int(case["mix"])))
    ns = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"])).astype(int)
    shapes = [("sphere", "ellipsoid", "torus")[s] for s in rng.integers(0, 3, case["count"])]
    return [(int(n), s) for n, s in zip(ns, shapes)]


# ---------------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        pts = [_points(s, n, seed * 1009 + i)[0] for i, (n, s) in enumerate(sizes)]
        pipe = BatchPipeline([(n, case["k"], case["nrhs"]) for n, _ in sizes], prec=PREC[case["prec"]], precond=2,
                             rtol=RTOL)
        return dict(kind=kind, pipe=pipe, pts=pts, f=[_rhs(p, case["nrhs"]) for p in pts])
    n, k = case["n"], case["k"]
    p, flags = _points(case["shape"], n, seed)
    st = dict(kind=kind, n=n, k=k, pts=p)
    if kind != "knn":
        st["prec"] = PREC[case["prec"]]
    if kind == "cloud":
        st["f"] = _rhs(p, case["nrhs"])
        st["pipe"] = Pipeline(n, k, case["nrhs"], prec=st["prec"], precond=2, rtol=RTOL)
    elif kind == "open":
        st["flags"] = flags
        st["f"] = (3.0 * p[:, 2]).contiguous()
    elif kind in ("assemble", "spmv", "solve"):
        st["nbr"], st["order"] = api.knn(p, k, want_order=True)
        if kind != "assemble":
            st["op"] = api.assemble(p, st["nbr"], prec=st["prec"], order=st["order"])
        if kind == "spmv":
            st["mode"] = {"f64": api.SPMV_F64, "f32": api.SPMV_F32, "hilo": api.SPMV_F64_HILO}[case["mode"]]
            st["x"] = _vectors(n, case["nrhs"], seed, torch.float32 if case["mode"] == "f32" else torch.float64)
        if kind == "solve":
            st["f"] = _rhs(p, case["nrhs"])
            st["precond"] = case["precond"]
            st["amg"] = api.amg_setup(st["op"]) if case["precond"] == 2 else None
    return st


def _weights(op):
    """The operator's FP64 weights in the stored layout (hi + lo in the mixed format)."""
    used = api.n_padded(op.n) * (op.k + 1)
    if op.prec == api.FP64:
        return op.val[:used]
    return op.val[:used].double() + op.val_lo[:used]


def run(st):
    kind = st["kind"]
    if kind == "rows":
        nbr, order = api.knn(st["pts"], st["k"], want_order=True)
        op = api.assemble(st["pts"], nbr, prec=st["prec"], order=order)
        lx = api.spmv(op, st["pts"][order.long()], sigma=0.0, alpha=-1.0)
        return dict(nbr=nbr, order=order, weights=_weights(op), lx=lx)
    if kind == "knn":
        nbr, order = api.knn(st["pts"], st["k"], want_order=True)
        return dict(nbr=nbr, order=order)
    if kind == "assemble":
        op = api.assemble(st["pts"], st["nbr"], prec=st["prec"], order=st["order"])
        return dict(weights=_weights(op), col=op.col[: api.n_padded(op.n) * op.k], h=op.h, status=op.status,
                    bad_rows=op.bad_rows)
    if kind == "spmv":
        return api.spmv(st["op"], st["x"], mode=st["mode"])
    if kind == "solve":
        res = api.solve(st["op"], st["f"], rtol=RTOL, precond=st["precond"], amg=st["amg"])
        return dict(u=res.u, status=max(res.status))
    if kind == "open":
        nbr, order = api.knn(st["pts"], st["k"], want_order=True)
        op = api.assemble(st["pts"], nbr, prec=st["prec"], order=order)
        zeroed = api.dirichlet_rows(op, st["flags"])
        res = api.solve(op, st["f"], rtol=RTOL, precond=2)
        return dict(u=res.u, status=max(res.status), zeroed=zeroed, nbr=nbr, order=order)
    if kind == "cloud":
        st["pipe"].run(st["pts"], st["f"])
        return dict(u=st["pipe"].u, nbr=st["pipe"].nbr, order=st["pipe"].order)
    st["pipe"].run(st["pts"], st["f"])
    return dict(u=[s.u for s in st["pipe"].slots], nbr=[s.nbr for s in st["pipe"].slots])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        per = [work(dict(case, kind="cloud", n=n)) for n, _ in _batch_sizes(case)]
        return dict(bytes=sum(w["bytes"] for w in per), flops=sum(w["flops"] for w in per))
    n, k = case["n"], case["k"]
    q = case.get("nrhs", 1)
    wide = 8.0 * (k + 1)                     # a row's weights, FP64 or hi + lo
    points, table, cols = 24.0 * n, 4.0 * n * k, 4.0 * n * k
    if kind == "knn":
        return dict(bytes=points + table + 4.0 * n, flops=8.0 * n * k)
    if kind == "assemble":
        return dict(bytes=points + table + 4.0 * n + wide * n + cols + 9.0 * n, flops=n * (90.0 * (k + 1) + 300.0))
    if kind == "rows":
        return dict(bytes=points + table + 4.0 * n + wide * n + cols + 48.0 * n,
                    flops=n * (98.0 * (k + 1) + 300.0))
    if kind == "spmv":
        esz = 4.0 if case["mode"] == "f32" else 8.0
        return dict(bytes=n * (esz * (k + 1) + 4.0 * k + 2.0 * q * esz), flops=2.0 * n * (k + 1) * q)
    if kind == "solve":
        return dict(bytes=n * (wide + 4.0 * k + 16.0 * q), flops=2.0 * n * (k + 1) * q)
    # points to solution: the cloud and f in, neighbours and u out, the operator formed and read once
    return dict(bytes=points + table + 16.0 * n * q + 2.0 * (wide * n + cols),
                flops=n * (98.0 * (k + 1) + 300.0) + 2.0 * n * (k + 1) * q)


# ---------------------------------------------------------------------------------------------------
# The same results in plain torch, FP64
# ---------------------------------------------------------------------------------------------------
def _nearest(p, q_idx, cand, k):
    """The k nearest of each query's candidates (padded with -1), ascending (distance, index)."""
    d = p[cand.clamp(min=0)] - p[q_idx][:, None]
    d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    d2 = torch.where((cand < 0) | (cand == q_idx[:, None]), math.inf, d2)
    v, at = torch.topk(d2, min(k + 4, d2.shape[1]), dim=1, largest=False)
    j = torch.gather(cand, 1, at)
    j, by = torch.sort(j, dim=1)
    v, by = torch.sort(torch.gather(v, 1, by), dim=1, stable=True)
    return torch.gather(j, 1, by)[:, :k], v[:, :k]


def _knn_exact(p, k):
    n = p.shape[0]
    every = torch.arange(n, device=p.device)
    if n <= 24_000:
        return torch.cat([_nearest(p, q, every[None].expand(len(q), n), k)[0] for q in every.split(1024)])
    lo = p.min(0).values
    _, v = _nearest(p, every[:: n // 64], every[None].expand(len(every[:: n // 64]), n), k)
    s = 1.5 * float(v[:, -1].max().sqrt())
    while True:
        c = ((p - lo) / s).long() + 1
        dims = c.max(0).values + 2
        key = (c[:, 0] * dims[1] + c[:, 1]) * dims[2] + c[:, 2]
        key, who = torch.sort(key)
        step = torch.tensor([-1, 0, 1], device=p.device)
        off = torch.cartesian_prod(step, step, step)
        off = (off[:, 0] * dims[1] + off[:, 1]) * dims[2] + off[:, 2]
        out, worst = torch.empty(n, k, dtype=torch.int64, device=p.device), 0.0
        for rows in torch.arange(n, device=p.device).split(8192):  # rows in cell order
            near = key[rows][:, None] + off
            a, b = torch.searchsorted(key, near), torch.searchsorted(key, near, right=True)
            width = max(1, int((b - a).max()))
            at = a[..., None] + torch.arange(width, device=p.device)
            cand = torch.where(at < b[..., None], who[at.clamp(max=n - 1)], -1).reshape(len(rows), -1)
            out[who[rows]], v = _nearest(p, who[rows], cand, k)
            worst = max(worst, float(v[:, -1].max()))
        if math.sqrt(worst) <= s:
            return out
        s *= 1.5


def _rows_exact(p, nbr):
    """(weights [n][k+1] with the point itself first, h), mean distance of the 6 nearest as the grid spacing."""
    ws, hs = [], []
    for at in torch.arange(p.shape[0], device=p.device).split(16_384):
        d = p[nbr[at]] - p[at][:, None]
        e = d - d.mean(1, keepdim=True)
        _, axes = torch.linalg.eigh(e.transpose(1, 2) @ e)
        h = d[:, :6].norm(dim=2).mean(1)
        loc = (d @ axes) / h[:, None, None]           # columns: normal, middle, largest
        loc = torch.cat([torch.zeros_like(loc[:, :1]), loc], 1)
        zeta, eta, xi = loc.unbind(2)
        v = torch.stack([torch.ones_like(xi), xi, eta, xi * xi, xi * eta, eta * eta], 2)
        gram = v.transpose(1, 2) @ v
        a = torch.linalg.solve(gram, v.transpose(1, 2) @ zeta[..., None])[..., 0]
        zx, zy = a[:, 1], a[:, 2]
        zxx, zxy, zyy = 2 * a[:, 3] / h, a[:, 4] / h, 2 * a[:, 5] / h
        w = 1 + zx * zx + zy * zy
        g11, g12, g22 = (1 + zy * zy) / w, -zx * zy / w, (1 + zx * zx) / w
        hs_ = g11 * zxx + 2 * g12 * zxy + g22 * zyy
        c = torch.stack([2 * (g11 + g22), -hs_ * zx / w * h, -hs_ * zy / w * h, 2 * g11, 2 * g12, 2 * g22], 1)
        y = (v @ torch.linalg.solve(gram, c[..., None]))[..., 0]
        y[:, 0] -= c[:, 0]
        ws.append(y / (h * h)[:, None])
        hs.append(h)
    return torch.cat(ws), torch.cat(hs)


def _order_exact(p):
    lo = p.min(0).values
    e = (p.max(0).values - lo).max()
    t = torch.clamp((p - lo) * (2097152.0 / e), 0.0, 2097151.0).long()
    key = torch.zeros(p.shape[0], dtype=torch.int64, device=p.device)
    for b in range(21):
        for a in range(3):
            key |= ((t[:, a] >> b) & 1) << (3 * b + a)
    return torch.sort(key, stable=True).indices


def _stored(w):
    """[n][m] rows -> the stored layout: slices of 32 rows, slot by slot, zero rows at the end."""
    n, m = w.shape
    full = torch.zeros((n + SLICE - 1) // SLICE * SLICE, m, dtype=w.dtype, device=w.device)
    full[:n] = w
    return full.reshape(-1, SLICE, m).transpose(1, 2).reshape(-1)


def _solve_exact(w, nbr, f, flags=None):
    n = w.shape[0]
    a = torch.zeros(n, n, dtype=torch.float64, device=w.device)
    a.scatter_(1, nbr, -w[:, 1:])
    a.diagonal().sub_(w[:, 0])
    if flags is not None:
        a[flags.bool()] = 0.0
    a.diagonal().add_(1.0)
    f2 = f.reshape(n, -1)
    lu, piv = torch.linalg.lu_factor(a)
    u = torch.linalg.lu_solve(lu, piv, f2)
    u = u + torch.linalg.lu_solve(lu, piv, f2 - a @ u)
    return u.reshape(f.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "knn":
        return None  # whole numbers
    if kind == "batch":
        out = []
        for i, (n, s) in enumerate(_batch_sizes(case)):
            if n > DENSE_MAX_BATCH:
                out.append(None)
                continue
            p = _points(s, n, seed * 1009 + i)[0]
            nbr = _knn_exact(p, case["k"])
            out.append(_solve_exact(_rows_exact(p, nbr)[0], nbr, _rhs(p, case["nrhs"])))
        return dict(u=out, nbr=[None] * len(out))
    n, k = case["n"], case["k"]
    if kind in ("solve", "cloud", "open") and n > DENSE_MAX:
        return None
    p, flags = _points(case["shape"], n, seed)
    nbr = _knn_exact(p, k)
    w, h = _rows_exact(p, nbr)
    if kind == "solve":
        return dict(u=_solve_exact(w, nbr, _rhs(p, case["nrhs"])), status=None)
    if kind == "cloud":
        return dict(u=_solve_exact(w, nbr, _rhs(p, case["nrhs"])), nbr=None, order=None)
    if kind == "open":
        return dict(u=_solve_exact(w, nbr, 3.0 * p[:, 2], flags), status=None, zeroed=None, nbr=None,
                    order=None)
    order = _order_exact(p)
    if kind == "assemble":
        return dict(weights=_stored(w[order]), col=None, h=h, status=None, bad_rows=None)
    if kind == "rows":
        lx = w[:, :1] * p + (w[:, 1:, None] * p[nbr]).sum(1)
        return dict(nbr=None, order=None, weights=_stored(w[order]), lx=lx[order])
    x = _vectors(n, case["nrhs"], seed, torch.float32 if case["mode"] == "f32" else torch.float64).double()
    place = torch.empty_like(order)
    place[order] = torch.arange(n, device=order.device)
    w, nbr = w[order], place[nbr[order]]
    lx = w[:, :1] * x
    for s in range(k):
        lx += w[:, s + 1: s + 2] * x[nbr[:, s]]
    return x - lx
