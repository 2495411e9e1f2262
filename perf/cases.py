"""The work that users of this framework have it do, as measured cases.

Each case is one call (or one short sequence of calls) of the public Python
binding on inputs drawn from a seed: stochastic trace estimation workloads of
the sizes that the repository's configurations, tests and benchmark use, and
generic sizes around them.  The inputs (matrices, training data) are made here
with torch on the GPU, in the CSR form that the binding takes.

`exact` gives the same outputs in 64-bit arithmetic with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_10516_gb300 import mlt

DEV = "cuda"


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The paper's log-determinant table on a small SPD matrix: three levels
        # of the multilevel estimator in one ragged call, FP64.  The smallest
        # calls are of this kind, many in a row, where latency counts.
        {"name": "logdet_grid64", "kind": "moments", "matrix": "grid2d", "size": 64, "precision": "fp64",
         "n1": 256, "d1": 8, "n2": 64, "d2": 32, "n3": 16, "d3": 128, "reorder": False, "tune": False},
        # The nuclear norm of a small directed graph (10,617 vertices, 72,176
        # edges: the size of the paper's automated-level study): X^T X by two
        # products a step, two levels, FP64.
        {"name": "nuclear_graph10k", "kind": "moments", "matrix": "gram", "size": 10617, "ncols": 10617,
         "nnz": 72176, "precision": "fp64", "n1": 400, "d1": 20, "n2": 60, "d2": 67, "n3": 10, "d3": 300,
         "reorder": False, "tune": False},
        # The streaming operator at its largest: a 7-point diffusion stencil on
        # a 100^3 grid, FP32, 128 probes to degree 128.
        {"name": "stencil100_fp32", "kind": "moments", "matrix": "diffusion", "size": 100, "precision": "fp32",
         "n1": 0, "d1": 0, "n2": 0, "d2": 0, "n3": 128, "d3": 128, "reorder": False, "tune": True},
        # The Estrada index on the scale-22 graph, the largest workload:
        # FP64-class moments in double-float, operator relabelled by degree.
        {"name": "estrada_rmat22_df64", "kind": "moments", "matrix": "rmat", "size": 22, "precision": "df64",
         "n1": 0, "d1": 0, "n2": 0, "d2": 0, "n3": 128, "d3": 64, "reorder": True, "tune": True},
        # The moment call behind the learned level at scale 20: many probes at
        # the 16 input moments, few above, FP32.
        {"name": "learned_rmat20_fp32", "kind": "moments", "matrix": "rmat", "size": 20, "precision": "fp32",
         "n1": 1000, "d1": 15, "n2": 17, "d2": 64, "n3": 2, "d3": 128, "reorder": True, "tune": True},
        # The nuclear norm of a 2^18 x 2^16 sparse matrix, FP32, 512 probes.
        {"name": "nuclear_2e18_fp32", "kind": "moments", "matrix": "gram", "size": 262144, "ncols": 65536,
         "nnz": 1717987, "precision": "fp32", "n1": 0, "d1": 0, "n2": 0, "d2": 0, "n3": 512, "d3": 128,
         "reorder": False, "tune": True},
        # Triangle counting on the scale-20 graph: exact integer moments of
        # 1024 probes and the control-variate estimate.
        {"name": "triangles_rmat20", "kind": "triangles", "size": 20, "probes": 1024},
        # Many SPD operators of uneven sizes and ragged levels in one persistent
        # batch (one graph launch), FP64.
        {"name": "batch16_fp64", "kind": "batch", "count": 16, "smin": 10, "smax": 72, "precision": "fp64"},
        # The whole call from host arrays: handle, interval, multilevel
        # estimate with given levels, handle released.
        {"name": "estimate_from_host", "kind": "estimate", "size": 48, "n1": 200, "d1": 6, "n2": 30, "d2": 24,
         "n3": 6, "d3": 96, "precision": "fp64"},
        # The spectrum interval of the scale-20 graph by Lanczos, which every
        # Estrada or nuclear-norm run asks for first.
        {"name": "interval_rmat20", "kind": "interval", "matrix": "rmat", "size": 20, "steps": 40},
        # Hutch++ on the Estrada index at scale 18: a 64-column sketch in FP32,
        # orthogonalised, and 64 deflated probes in double-float.
        {"name": "hutchpp_rmat18", "kind": "hutchpp", "size": 18, "s": 64, "g": 64, "degree": 64,
         "precision": "df64"},
        # Training of the learned level's network on 2^14 probes' features: the
        # gradient of the whole set, a few epochs of minibatches, predictions.
        {"name": "network_2e14", "kind": "network", "samples": 16384, "batch": 2048, "epochs": 5},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _levels(rng, nmax, dmax):
    d1 = rng.randint(4, 20)
    d2 = rng.randint(d1 + 1, 70)
    d3 = rng.randint(d2 + 1, dmax)
    n3 = _log_uniform(rng, 2, max(3, nmax // 16))
    return {"n1": _log_uniform(rng, 16, nmax), "d1": d1, "n2": _log_uniform(rng, 4, max(5, nmax // 4)), "d2": d2,
            "n3": n3, "d3": d3}


def draw(rng):
    """One more case of the same kinds, sizes spread over their ranges."""
    while True:
        kind = rng.choice(["grid2d", "diffusion", "diffusion", "rmat", "rmat", "gram", "gram", "triangles", "batch",
                           "estimate", "interval", "hutchpp", "network"])
        prec = rng.choice(["fp64", "fp32", "df64"])
        if kind == "grid2d":
            c = {"kind": "moments", "matrix": "grid2d", "size": _log_uniform(rng, 12, 300), "precision": prec,
                 "reorder": False, "tune": False, **_levels(rng, 400, 256)}
        elif kind == "diffusion":
            c = {"kind": "moments", "matrix": "diffusion", "size": _log_uniform(rng, 8, 110), "precision": prec,
                 "reorder": False, "tune": rng.random() < 0.5, **_levels(rng, 256, 192)}
        elif kind == "rmat":
            c = {"kind": "moments", "matrix": "rmat", "size": rng.randint(10, 21), "precision": prec,
                 "reorder": rng.random() < 0.7, "tune": rng.random() < 0.5, **_levels(rng, 400, 128)}
        elif kind == "gram":
            nr = _log_uniform(rng, 300, 300000)
            nc = _log_uniform(rng, max(100, nr // 8), nr)
            c = {"kind": "moments", "matrix": "gram", "size": nr, "ncols": nc, "nnz": int(nr * rng.uniform(3, 20)),
                 "precision": prec, "reorder": False, "tune": rng.random() < 0.5, **_levels(rng, 400, 256)}
        elif kind == "triangles":
            c = {"kind": "triangles", "size": rng.randint(8, 20), "probes": _log_uniform(rng, 10, 1500)}
        elif kind == "batch":
            smin = rng.randint(6, 16)
            c = {"kind": "batch", "count": rng.randint(2, 24), "smin": smin, "smax": rng.randint(smin + 4, 72),
                 "precision": prec}
        elif kind == "estimate":
            c = {"kind": "estimate", "size": _log_uniform(rng, 8, 90), "precision": prec, **_levels(rng, 256, 128)}
        elif kind == "interval":
            c = {"kind": "interval", "matrix": rng.choice(["rmat", "diffusion", "gram"]), "steps": rng.randint(20, 50)}
            if c["matrix"] == "rmat":
                c["size"] = rng.randint(10, 21)
            elif c["matrix"] == "diffusion":
                c["size"] = _log_uniform(rng, 8, 110)
            else:
                c["size"] = _log_uniform(rng, 300, 300000)
                c["ncols"] = max(100, int(c["size"] * rng.uniform(0.125, 1.0)))
                c["nnz"] = int(c["size"] * rng.uniform(3, 20))
        elif kind == "network":
            c = {"kind": "network", "samples": _log_uniform(rng, 200, 1 << 17), "batch": _log_uniform(rng, 64, 8192),
                 "epochs": rng.randint(1, 8)}
        else:
            c = {"kind": "hutchpp", "size": rng.randint(10, 19), "s": rng.randint(8, 64), "g": rng.randint(8, 64),
                 "degree": rng.randint(16, 80), "precision": rng.choice(["fp64", "df64"])}
        if _cost(c) <= 0.9 * _cost(listed()[3]):
            return c


# ---------------------------------------------------------------------------
# sizes, costs, work
# ---------------------------------------------------------------------------

VB = {"fp64": 8, "fp32": 4, "df64": 8}       # bytes of a vector entry


def _shape(c):
    """(dimension, stored entries, entry bytes, extra rows of a Gram step)."""
    m = c.get("matrix", {"triangles": "rmat", "hutchpp": "rmat", "estimate": "diffusion"}.get(c["kind"]))
    s = c["size"]
    if m == "grid2d":
        return s * s, 5 * s * s - 4 * s, 12, 0
    if m == "diffusion":
        return s ** 3, 7 * s ** 3 - 6 * s * s, 12, 0
    if m == "rmat":
        return 1 << s, int(30.5 * (1 << s)) if s >= 18 else int(24 * (1 << s)), 4, 0
    return c["ncols"], c["nnz"], 12, s


def _degrees(c):
    return np.concatenate([np.full(c["n%d" % k], c["d%d" % k], dtype=np.int32) for k in (1, 2, 3)])


def _batch_sizes(c):
    """Grid edges from smin to smax, evenly over the number of matrices."""
    n = c["count"]
    return [int(round(c["smin"] + (c["smax"] - c["smin"]) * i / max(1, n - 1))) for i in range(n)]


def _batch_degrees(i):
    """Ragged levels of matrix i: three or four levels of degree 16 to 256."""
    parts = [(24 + 5 * (i % 4), 16), (8 + i % 5, 64)]
    if i % 2:
        parts.append((4, 128))
    parts.append((2, 256))
    return np.concatenate([np.full(n, d, dtype=np.int32) for n, d in parts])


def _recurrence(d, nnz, eb, extra, degrees, vb):
    """Bytes and flops of a ragged doubling recurrence.  Where matrix and live
    vectors fit on the chip, the matrix counts once; else each step streams the
    matrix and reads two vectors of each live probe and writes one."""
    steps = (degrees.astype(np.int64) + 1) // 2
    gram = 2 if extra else 1
    matrix = gram * (eb * nnz + 8 * d) + 8 * extra
    flops = float(steps.sum()) * (2 * nnz * gram + 8 * d)
    out = 8.0 * len(degrees) * (int(degrees.max()) + 1)
    if matrix + 2 * d * vb * len(degrees) <= 100e6:
        return matrix + out, flops
    launches = int(steps.max())
    return float(launches) * matrix + float(steps.sum()) * (3 * d + 2 * extra) * vb + out, flops


def work(c):
    kind = c["kind"]
    if kind == "batch":
        b = f = 0.0
        for i, s in enumerate(_batch_sizes(c)):
            x, y = _recurrence(s ** 3, 7 * s ** 3, 12, 0, _batch_degrees(i), VB[c["precision"]])
            b += x
            f += y
        return {"bytes": b, "flops": f}
    if kind == "network":       # forward and backward of the 16-128-128-1 network, gradient pass, epochs, forward
        n, par = c["samples"], 18817
        passes = 1 + c["epochs"]
        steps = c["epochs"] * -(-n // c["batch"])
        return {"bytes": 4.0 * (17 * n + 3 * par + n), "flops": 2.0 * 18560 * n * (3 * passes + 1) + 10.0 * par * steps}
    d, nnz, eb, extra = _shape(c)
    if kind == "moments" or kind == "estimate":
        b, f = _recurrence(d, nnz, eb, extra, _degrees(c), VB[c["precision"]])
        return {"bytes": b, "flops": f}
    if kind == "triangles":     # the graph once, one 256-probe block of signs and row sums a pass
        blocks = -(-c["probes"] // 256)
        return {"bytes": float(blocks) * (6 * nnz + 16 * d + 2 * 256 * d), "flops": 4.0 * nnz * c["probes"]}
    if kind == "interval":      # one product and three vectors a step
        g = 2 if extra else 1
        return {"bytes": float(c["steps"]) * (g * (eb * nnz + 8 * d) + 24 * (d + extra)),
                "flops": float(c["steps"]) * (2 * nnz * g + 10 * d)}
    # hutchpp: the sketch's applications in FP32, then the moments of Q and the probes
    n = c["degree"]
    mv = n * c["s"] + (n // 2) * (c["s"] + c["g"])
    width = 3 * 4 * n * c["s"] + 3 * 8 * (n // 2) * (c["s"] + c["g"])
    return {"bytes": 4.0 * nnz * 2 * n + float(d) * width, "flops": float(mv) * (2 * nnz + 8 * d)}


def _cost(c):
    """Rough time, for keeping drawn cases below the largest listed one."""
    if c["kind"] == "network":      # many small steps in a row
        return 30e-6 * c["epochs"] * (c["samples"] / c["batch"] + 1)
    w = work(c)
    slow = 8.0 if c.get("precision") == "fp64" or c["kind"] == "interval" else 1.0
    return w["bytes"] / 4e12 + slow * w["flops"] / 8e12


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Csr:
    """CSR arrays in the form mlt.Matrix takes (CUDA tensors, or numpy)."""

    def __init__(self, nrows, ncols, rowptr, col, val):
        self.nrows, self.ncols = nrows, ncols
        self.rowptr, self.col, self.val = rowptr, col, val
        self.nnz = int(col.shape[0])

    def host(self):
        return _Csr(self.nrows, self.ncols, self.rowptr.cpu().numpy(), self.col.cpu().numpy(),
                    None if self.val is None else self.val.cpu().numpy())


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _rowptr(counts):
    p = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=p[1:])
    return p


def _from_keys(key, nrows, ncols, val=None):
    r = torch.div(key, ncols, rounding_mode="floor")
    counts = torch.bincount(r, minlength=nrows)
    return _Csr(nrows, ncols, _rowptr(counts), (key - r * ncols).to(torch.int32), val)


def _rmat(scale, seed):
    """Symmetric 0/1 adjacency of an R-MAT graph, edge factor 16, (a, b, c) =
    (0.57, 0.19, 0.19), no self-loops or duplicates."""
    g = _gen(seed)
    n, m = 1 << scale, 16 << scale
    keys = []
    for s in range(0, m, 1 << 24):
        e = min(m, s + (1 << 24)) - s
        u = torch.zeros(e, dtype=torch.int64, device=DEV)
        v = torch.zeros(e, dtype=torch.int64, device=DEV)
        for _ in range(scale):
            r = torch.rand(e, generator=g, device=DEV)
            u = (u << 1) | (r >= 0.76)
            v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        ok = u != v
        u, v = u[ok], v[ok]
        keys += [u * n + v, v * n + u]
    key = torch.unique(torch.cat(keys))
    return _from_keys(key, n, n)


def _grid2d(s):
    """5-point Dirichlet Laplacian on an s x s grid plus 0.1 I."""
    i = torch.arange(s * s, device=DEV)
    return _stencil(i, [(i % s, 1, s), (torch.div(i, s, rounding_mode="floor"), s, s)],
                    lambda cell, nb: torch.full_like(cell, -1.0, dtype=torch.float64), None, 0.1)


def _stencil(i, axes, off, kappa, shift):
    """Rows i with neighbours at +-stride along each axis; kappa None: the
    constant diagonal 2 x axes + shift, else harmonic means of kappa."""
    d = i.numel()
    diag = torch.full((d,), float(shift), dtype=torch.float64, device=DEV)
    if kappa is None:
        diag += 2.0 * len(axes)
    keys, vals = [], []
    for x, stride, n in axes:
        for sgn in (-1, 1):
            ok = (x > 0) if sgn < 0 else (x < n - 1)
            nb = (i + sgn * stride).clamp_(0, d - 1)
            if kappa is None:
                face = torch.ones(d, dtype=torch.float64, device=DEV)
            else:
                face = torch.where(ok, 2.0 * kappa * kappa[nb] / (kappa + kappa[nb]), kappa)
                diag += face
            keys.append((i * d + nb)[ok])
            vals.append(-face[ok])
    keys.append(i * d + i)
    vals.append(diag)
    key, order = torch.sort(torch.cat(keys))
    return _from_keys(key, d, d, torch.cat(vals)[order])


def _diffusion(s, seed, shift):
    """7-point operator on an s^3 grid, lognormal cell coefficients (sigma 1),
    harmonic face means, Dirichlet boundary, plus shift I."""
    i = torch.arange(s ** 3, device=DEV)
    kappa = torch.exp(torch.randn(s ** 3, generator=_gen(seed), device=DEV, dtype=torch.float64))
    axes = [(i % s, 1, s), (torch.div(i, s, rounding_mode="floor") % s, s, s),
            (torch.div(i, s * s, rounding_mode="floor"), s * s, s)]
    return _stencil(i, axes, None, kappa, shift)


def _sparse_gaussian(nr, nc, nnz, seed):
    """X with about nnz uniform distinct positions and N(0, 1) values."""
    g = _gen(seed)
    key = torch.unique(torch.randint(0, nr * nc, (nnz,), generator=g, device=DEV, dtype=torch.int64))
    return _from_keys(key, nr, nc, torch.randn(key.numel(), generator=g, device=DEV, dtype=torch.float64))


def _torch_csr(m, dtype=torch.float64):
    val = torch.ones(m.nnz, dtype=dtype, device=DEV) if m.val is None else m.val.to(dtype)
    return torch.sparse_csr_tensor(m.rowptr.to(torch.int32), m.col, val, size=(m.nrows, m.ncols))


def _transpose(m):
    rows = torch.repeat_interleave(torch.arange(m.nrows, device=DEV), m.rowptr.diff())
    key, order = torch.sort(m.col.to(torch.int64) * m.nrows + rows)
    return _from_keys(key, m.ncols, m.nrows, None if m.val is None else m.val[order])


def _power_radius(mul, d, seed, steps):
    """Norm estimate of a symmetric operator by power iteration on a block of four."""
    x = torch.randn((d, 4), generator=_gen(seed + 1), device=DEV, dtype=torch.float64)
    est = 0.0
    for _ in range(steps):
        x /= torch.linalg.vector_norm(x, dim=0).clamp_min(1e-300)
        x = mul(x)
        est = torch.linalg.vector_norm(x, dim=0).max()
    return float(est)


class _Problem:
    """A matrix, its interval and scale as a user has them before the call."""

    def __init__(self, kind, c, seed):
        self.scale, self.gram, self.at = 1.0, False, None
        if kind == "grid2d":
            self.m = _grid2d(c["size"])
            self.a, self.b = 0.1, 8.1
        elif kind == "diffusion":
            self.m = _diffusion(c["size"], seed, 0.05 + (seed % 97) / 100.0)
            dense_row = torch.zeros(self.m.nrows, dtype=torch.float64, device=DEV)
            rows = torch.repeat_interleave(torch.arange(self.m.nrows, device=DEV), self.m.rowptr.diff())
            dense_row.index_add_(0, rows, self.m.val.abs())
            self.a, self.b = 0.04, float(dense_row.max()) * 1.000001
        elif kind == "rmat":
            self.m = _rmat(c["size"], seed)
            t = _torch_csr(self.m, torch.float32)
            radius = _power_radius(lambda x: (t @ x.float()).double(), self.m.nrows, seed, 40)
            self.scale = 10.0 / (1.02 * radius)
            self.a, self.b = -10.0, 10.0
        else:
            self.m = _sparse_gaussian(c["size"], c["ncols"], c["nnz"], seed)
            self.gram = True
            x, xt = _torch_csr(self.m), _torch_csr(_transpose(self.m))
            self.a, self.b = 0.0, 1.15 * _power_radius(lambda v: xt @ (x @ v), self.m.ncols, seed, 60)
        self.dim = self.m.ncols

    def operator(self):
        """The scaled, unmapped operator in 64 bits, as a function of a block."""
        t = _torch_csr(self.m)
        if self.gram:
            tt = _torch_csr(_transpose(self.m))
            return lambda v: tt @ (t @ v)
        return lambda v: (t @ v) * self.scale

    def mapped(self):
        op = self.operator()
        al, be = 2.0 / (self.b - self.a), -(self.a + self.b) / (self.b - self.a)
        return lambda v: al * op(v) + be * v


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _probe_seed(seed):
    return int(seed) * 2654435761 % (1 << 31) + 3


def _samples(c, seed):
    """Standardised features (moments of a probe, which share a common factor)
    and a smooth target of them, FP32."""
    g = _gen(seed)
    n = c["samples"]
    mix = torch.randn((16, 16), generator=g, device=DEV) / 4.0
    x = torch.randn((n, 16), generator=g, device=DEV) @ mix + torch.randn((n, 1), generator=g, device=DEV)
    x = (x - x.mean(0)) / x.std(0)
    t = torch.tanh(x[:, 0]) + 0.5 * x[:, 1] * x[:, 2] + 0.1 * torch.randn(n, generator=g, device=DEV)
    return x.contiguous(), ((t - t.mean()) / t.std()).contiguous()


def _params(c, seed):
    """The starting weights (W1, b1, W2, b2, w3, b3) a program brings: He-scaled normals, zero biases."""
    g = _gen(seed + 5)
    parts = [torch.randn(2048, generator=g, device=DEV) * math.sqrt(2 / 16), torch.zeros(128, device=DEV),
             torch.randn(16384, generator=g, device=DEV) * math.sqrt(2 / 128), torch.zeros(128, device=DEV),
             torch.randn(128, generator=g, device=DEV) * math.sqrt(1 / 128), torch.zeros(1, device=DEV)]
    return torch.cat(parts)


def _tune(handle, c):
    """A program that makes many calls on a handle tunes it once."""
    if c.get("tune"):
        mlt.mlt_autotune(handle, c["precision"], 4)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": _probe_seed(seed)}
    if kind == "batch":
        st["mats"], jobs = [], []
        for i, s in enumerate(_batch_sizes(case)):
            p = _Problem("diffusion", {"size": s}, seed * 100 + i)
            deg = _batch_degrees(i)
            M = mlt.Matrix(p.m)
            out = torch.zeros((deg.size, int(deg.max()) + 1), dtype=torch.float64, device=DEV)
            st["mats"].append(M)
            jobs.append({"matrix": M.handle, "a": p.a, "b": p.b, "seed": st["seed"] + i, "probe_offset": 0,
                         "degrees": deg, "out": out, "group_width": 0})
        st["outs"] = [j["out"] for j in jobs]
        st["batch"] = mlt.Batch(jobs, precision=case["precision"])
        return st
    if kind == "estimate":
        p = _Problem("diffusion", case, seed)
        st["csr"] = p.m.host()
        return st
    if kind == "network":
        st["x"], st["t"] = (v.cpu().numpy() for v in _samples(case, seed))
        st["params"] = _params(case, seed).cpu().numpy()
        st["net"] = mlt.Surrogate(seed=st["seed"])
        return st
    p = _Problem(case.get("matrix", "rmat"), case, seed)
    st["p"] = p
    st["M"] = mlt.Matrix(p.m, gram=p.gram, scale=p.scale, reorder=bool(case.get("reorder")))
    if kind == "moments":
        st["deg"] = _degrees(case)
        # small results go to host memory, large runs keep them on the device
        if st["deg"].size * (int(st["deg"].max()) + 1) * p.dim > 1 << 32:
            st["out"] = torch.zeros((st["deg"].size, int(st["deg"].max()) + 1), dtype=torch.float64, device=DEV)
        else:
            st["out"] = np.zeros((st["deg"].size, int(st["deg"].max()) + 1))
        _tune(st["M"].handle, case)
    elif kind == "triangles":
        st["x"] = np.zeros((case["probes"], 3), dtype=np.int64)
    elif kind == "hutchpp":
        st["c"] = mlt.mlt_cheb_coeffs("exp", p.a, p.b, case["degree"])
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "moments":
        return st["M"].moments(st["p"].a, st["p"].b, st["seed"], 0, st["deg"], precision=c["precision"], out=st["out"])
    if kind == "triangles":
        est, se = st["M"].triangles(st["seed"], 0, c["probes"], True, st["x"])
        return {"x": st["x"], "estimate": est, "stderr": se}
    if kind == "batch":
        st["batch"].run(0)
        return st["outs"]
    if kind == "estimate":
        with mlt.Matrix(st["csr"]) as M:
            a, b = M.bounds()
            r = M.mlmc("log", a, b, c["d3"], seed=st["seed"], levels=[c["d1"], c["d2"], c["d3"]],
                       m=[c["n1"], c["n2"], c["n3"]], precision=c["precision"])
        return {"a": a, "b": b, "estimate": r["estimate"], "stderr": r["stderr"], "level_mean": r["level_mean"],
                "level_var": r["level_var"], "levels": r["levels"], "m": r["m"], "matvecs": r["matvecs"]}
    if kind == "network":
        net = st["net"]
        net.set_params(st["params"])
        loss, grad = net.loss_grad(st["x"], st["t"])
        last = net.train(st["x"], st["t"], c["epochs"], c["batch"], 1e-3)
        return {"loss": loss, "grad": grad, "last": last, "params": net.get_params(), "y": net.predict(st["x"])}
    if kind == "interval":
        a, b = mlt.mlt_spectrum_bounds(st["M"].handle, mlt.MLT_BOUNDS_LANCZOS, c["steps"], st["seed"])
        return {"a": a, "b": b}
    samples = np.zeros(c["g"])
    r = mlt.mlt_hutchpp_estimate(st["M"].handle, st["p"].a, st["p"].b, st["c"], st["seed"], 0, c["s"], c["g"],
                                 c["precision"], samples)
    return {"estimate": r.estimate, "std_error": r.std_error, "t_sketch": r.t_sketch, "t_rest": r.t_rest,
            "rank": r.rank, "samples": samples}


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------

def _i64(v):
    """A 64-bit pattern as a signed Python int."""
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _lsr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _signs(d, ids, seed):
    """Probe entries (d x len(ids), float64): the documented counter hash."""
    i = torch.arange(d, dtype=torch.int64, device=DEV)
    mix = _i64(seed * 0x9E3779B97F4A7C15)
    out = torch.empty((d, len(ids)), dtype=torch.float64, device=DEV)
    words = {}
    for k, p in enumerate(ids):
        q = p >> 6
        if q not in words:
            x = (i | (q << 32)) ^ mix
            x = (x ^ _lsr(x, 30)) * _i64(0xBF58476D1CE4E5B9)
            x = (x ^ _lsr(x, 27)) * _i64(0x94D049BB133111EB)
            words = {q: x ^ _lsr(x, 31)}
        out[:, k] = 1.0 - 2.0 * ((words[q] >> (p & 63)) & 1).double()
    return out


def _moments64(op, d, z, n):
    """mu_0 .. mu_n of the columns of z by the doubling identities."""
    mu = torch.zeros((z.shape[1], n + 1), dtype=torch.float64, device=DEV)
    mu[:, 0] = d
    if n == 0:
        return mu
    prev, cur = z, op(z)
    x0 = (cur * prev).sum(0)
    for k in range((n + 1) // 2):           # cur = V_{k+1}, prev = V_k
        if k > 0:
            prev, cur = cur, 2.0 * op(cur) - prev
        mu[:, 2 * k + 1] = x0 if k == 0 else 2.0 * (cur * prev).sum(0) - x0
        if 2 * k + 2 <= n:
            mu[:, 2 * k + 2] = 2.0 * (cur * cur).sum(0) - d
    return mu


def _ragged64(op, d, degrees, seed):
    out = torch.zeros((len(degrees), int(degrees.max()) + 1), dtype=torch.float64, device=DEV)
    width = max(1, min(128, int(6e9 / (8 * d))))
    for deg in sorted(set(degrees.tolist())):
        ids = [int(p) for p in np.nonzero(degrees == deg)[0]]
        for s in range(0, len(ids), width):
            part = ids[s:s + width]
            out[part, :deg + 1] = _moments64(op, d, _signs(d, part, seed), int(deg))
    return out


def _cheb64(f, a, b, n):
    x = np.cos(np.arange(n + 1) * np.pi / n)
    fx = f(0.5 * (b - a) * x + 0.5 * (a + b))
    w = np.ones(n + 1)
    w[0] = w[-1] = 0.5
    c = np.array([(2.0 / n) * np.sum(w * fx * np.cos(np.arange(n + 1) * k * np.pi / n)) for k in range(n + 1)])
    c[0] *= 0.5
    c[n] *= 0.5
    return c


def exact(case, seed):
    kind, ps = case["kind"], _probe_seed(seed)
    if kind == "batch":
        out = []
        for i, s in enumerate(_batch_sizes(case)):
            p = _Problem("diffusion", {"size": s}, seed * 100 + i)
            out.append(_ragged64(p.mapped(), p.dim, _batch_degrees(i), ps + i))
        return out
    if kind == "estimate":
        p = _Problem("diffusion", case, seed)
        m = p.m
        rows = torch.repeat_interleave(torch.arange(m.nrows, device=DEV), m.rowptr.diff())
        on = rows == m.col
        diag = torch.zeros(m.nrows, dtype=torch.float64, device=DEV).index_add_(0, rows[on], m.val[on])
        off = torch.zeros(m.nrows, dtype=torch.float64, device=DEV).index_add_(0, rows[~on], m.val[~on].abs())
        p.a, p.b = float((diag - off).min()), float((diag + off).max())
        deg = _degrees(case)
        mu = _ragged64(p.mapped(), p.dim, deg, ps).cpu().numpy()
        c = _cheb64(np.log, p.a, p.b, case["d3"])
        means, variances, q, lo, est, var = [], [], 0, -1, 0.0, 0.0
        for k in (1, 2, 3):
            n, hi = case["n%d" % k], case["d%d" % k]
            v = mu[q:q + n, lo + 1:hi + 1] @ c[lo + 1:hi + 1]
            q, lo = q + n, hi
            means.append(float(v.mean()))
            variances.append(float(v.var(ddof=1)))
            est += means[-1]
            var += variances[-1] / n
        return {"a": p.a, "b": p.b, "estimate": est, "stderr": math.sqrt(var), "level_mean": means,
                "level_var": variances, "levels": None, "m": None, "matvecs": None}
    if kind == "network":       # the loss and gradient at the given weights (the rest follows a rounded path)
        x, t = (v.double() for v in _samples(case, seed))
        w = _params(case, seed).double().requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = (w[i:j] for i, j in ((0, 2048), (2048, 2176), (2176, 18560), (18560, 18688),
                                                      (18688, 18816), (18816, 18817)))
        h = torch.relu(x @ w1.reshape(128, 16).T + b1)
        h = torch.relu(h @ w2.reshape(128, 128).T + b2)
        loss = ((h @ w3 + b3 - t) ** 2).mean()
        loss.backward()
        return {"loss": float(loss.detach()), "grad": w.grad, "last": None, "params": None, "y": None}
    p = _Problem(case.get("matrix", "rmat"), case, seed)
    d = p.dim
    if kind == "moments":
        return _ragged64(p.mapped(), d, _degrees(case), ps)
    if kind == "triangles":
        t = _torch_csr(p.m)
        xs = []
        for s in range(0, case["probes"], 64):
            z = _signs(d, list(range(s, min(case["probes"], s + 64))), ps)
            y = t @ z
            w = (t @ y).to(torch.int64)
            zi, yi = z.to(torch.int64), y.to(torch.int64)
            xs.append(torch.stack([(zi * yi).sum(0), (yi * yi).sum(0), (yi * w).sum(0)], 1))
        x = torch.cat(xs).cpu().numpy()
        m = x.shape[0]
        f = x.astype(np.longdouble)
        f = f - f.mean(0)
        s11, s12, s22 = (f[:, 0] ** 2).sum(), (f[:, 0] * f[:, 1]).sum(), (f[:, 1] ** 2).sum()
        r1, r2 = (f[:, 0] * f[:, 2]).sum(), (f[:, 1] * f[:, 2]).sum()
        det = s11 * s22 - s12 * s12
        a1, a2 = (s22 * r1 - s12 * r2) / det, (s11 * r2 - s12 * r1) / det
        mean = [np.longdouble(int(x[:, k].astype(object).sum())) / m for k in range(3)]
        est = (mean[2] - a2 * (mean[1] - p.m.nnz) - a1 * mean[0]) / 6
        res = ((f[:, 2] - a1 * f[:, 0] - a2 * f[:, 1]) ** 2).sum() / (m - 3)
        return {"x": x, "estimate": float(est), "stderr": float(np.sqrt(res / m) / 6)}
    if kind == "interval":
        op = p.operator()
        q = _signs(d, [0], ps) / math.sqrt(d)
        prev, bprev, al, be = torch.zeros_like(q), 0.0, [], []
        for _ in range(min(max(case["steps"], 2), d)):
            w = op(q)
            a = float((q * w).sum())
            w = w - a * q - bprev * prev
            b = math.sqrt(float((w * w).sum()))
            al.append(a)
            be.append(b)
            if not b > 1e-12 * (abs(a) + bprev):
                break
            prev, q, bprev = q, w / b, b
        n = len(al)
        th, S = np.linalg.eigh(np.diag(al) + np.diag(be[:n - 1], 1) + np.diag(be[:n - 1], -1))
        lo, hi = th[0] - abs(be[-1] * S[-1, 0]), th[-1] + abs(be[-1] * S[-1, -1])
        lo, hi = lo - 0.01 * abs(lo), hi + 0.01 * abs(hi)
        return {"a": max(lo, 1e-6 * hi) if p.gram else lo, "b": hi}
    # hutchpp
    op, n = p.mapped(), case["degree"]
    c = _cheb64(np.exp, p.a, p.b, n)
    S = _signs(d, list(range(case["s"])), ps)
    prev, cur = S, op(S)
    Y = c[0] * prev + c[1] * cur
    for k in range(2, n + 1):
        prev, cur = cur, 2.0 * op(cur) - prev
        Y += c[k] * cur
    Q, R = torch.linalg.qr(Y)
    if bool((R.diagonal().abs() < 1e-6 * R.diagonal().abs().max()).any()):
        return None
    G = _signs(d, list(range(case["s"], case["s"] + case["g"])), ps)
    G = G - Q @ (Q.T @ G)

    def forms(block):
        mu = _moments64(op, 1.0, block, n).cpu().numpy()
        sq = (block * block).sum(0).cpu().numpy()
        mu[:, 0] = sq
        mu[:, 2::2] += 1.0 - sq[:, None]
        return mu @ c

    t = float(forms(Q).sum())
    smp = forms(G)
    return {"estimate": t + float(smp.mean()), "std_error": float(smp.std(ddof=1) / math.sqrt(case["g"])),
            "t_sketch": t, "t_rest": float(smp.mean()), "rank": None, "samples": smp}
