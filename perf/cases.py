"""Performance cases of the node-aware SpMV library: what its users run, at the sizes they run it.

A case is a dict of plain values with a ``kind``:

* ``apply``  one napspmv_apply, or a napspmv_apply_n / napspmv_apply_ex chain of ``reps`` products;
* ``batch``  one napspmv_apply_batch over many small matrices (a step of the request server);
* ``cg``     a whole napspmv_cg_ir solve, or napspmv_cg without refinement;
* ``cgstep`` napspmv_cg_batch_init and _iterate over several solves (a step of the request server);
* ``plan``   napspmv_plan and the first product with it.

Matrices are those of ``paper_1612_08060_gb300.inputs``, made on the GPU here: 2D 5-point (``p2d``), 3D
7-point (``p3d``) and 2D Q1 9-point (``q1``) stencils, and the banded random matrix (``banded``).
"""
import math
import random

import numpy as np
import torch

from paper_1612_08060_gb300 import inputs
from paper_1612_08060_gb300 import napspmv as nap

DEV = "cuda"


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the smallest product: the 64 x 64 grid that the examples and the smoke test run
        dict(name="apply_2d_64", kind="apply", mat="p2d", side=64, n_p=16, ppn=4, reps=1, prec="f64", part="block", scale=1.0),
        # a power-like iteration on the 3D 7-point matrix: 100 chained products
        dict(name="chain_3d_128", kind="apply", mat="p3d", side=128, n_p=1024, ppn=16, reps=100, prec="f64", part="block", scale=1.0 / 16),
        # the smoother-like use of FP32-stored values on the 9-point matrix, 20 chained products
        dict(name="chain_q1_2048_f32", kind="apply", mat="q1", side=2048, n_p=4096, ppn=16, reps=20, prec="f32", part="block", scale=1.0 / 4),
        # the unstructured matrix of the benchmark, 10 chained products: the largest
        dict(name="chain_banded_2p23", kind="apply", mat="banded", n=1 << 23, n_p=8192, ppn=32, reps=10, prec="f64", part="block", scale=1.0 / 128),
        # one product on a medium unstructured matrix; no size divides another
        dict(name="apply_banded_1m", kind="apply", mat="banded", n=1_000_003, n_p=977, ppn=24, reps=1, prec="f64", part="block", scale=1.0),
        # FP32-stored values on a long-row matrix, uneven partition
        dict(name="chain_banded_3m_f32", kind="apply", mat="banded", n=3_141_593, n_p=3067, ppn=32, reps=10, prec="f32", part="block", scale=1.0 / 128),
        # the strided partition of the paper's unstructured runs, odd grid
        dict(name="apply_3d_101_strided", kind="apply", mat="p3d", side=101, n_p=503, ppn=16, reps=1, prec="f64", part="strided", scale=1.0),
        # a server step: products on many small matrices in one call
        dict(name="batch_32_small", kind="batch", count=32, n_lo=1000, n_hi=100_000, mix=7, prec="f64"),
        # a whole solve to 1e-10: FP32-valued CG inside FP64 refinement
        dict(name="cg_ir_3d_63", kind="cg", mat="p3d", side=63, n_p=122, ppn=16, refine=True),
        # a server step: 8 CG iterations for each of 16 small solves
        dict(name="cgstep_16_small", kind="cgstep", count=16, n_lo=1000, n_hi=100_000, mix=11, iters=8, prec="f32"),
        # a server step of a large solve: 64 CG iterations on its own
        dict(name="cgstep_2d_1300", kind="cgstep", count=1, n_lo=1_690_000, n_hi=1_690_000, mix=-2, iters=64, prec="f32"),
        # a new matrix: the plan and its first product
        dict(name="plan_3d_100", kind="plan", mat="p3d", side=100, n_p=488, ppn=16, prec="f32"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _partition(rng, n, lo, hi):
    """Processes of lo..hi rows each, and their number per node."""
    return max(1, min(n, int(round(n / _log(rng, lo, hi))))), rng.choice([4, 8, 12, 16, 16, 24, 32, 32])


def draw(rng):
    kind = rng.choices(["apply", "batch", "cg", "cgstep", "plan"], [10, 2, 2, 2, 1])[0]
    if kind == "apply":
        mat = rng.choice(["p2d", "p3d", "q1", "banded", "banded"])
        c = dict(kind=kind, mat=mat)
        if mat == "banded":
            c["n"] = int(_log(rng, 20_000, 1 << 23))
            n, (c["n_p"], c["ppn"]) = c["n"], _partition(rng, c["n"], 700, 1500)
            c["reps"], c["scale"] = rng.choice([1, 4, 10]), 1.0 / 128
        else:
            dim, lo, hi = {"p2d": (2, 32, 1414), "p3d": (3, 10, 128), "q1": (2, 48, 2048)}[mat]
            c["side"] = int(_log(rng, lo, hi))
            n = c["side"] ** dim
            c["n_p"], c["ppn"] = _partition(rng, n, 256, 2048)
            c["reps"], c["scale"] = rng.choice([1, 5, 20]), {"p2d": 1.0 / 8, "p3d": 1.0 / 16, "q1": 1.0 / 4}[mat]
        c["prec"] = rng.choice(["f64", "f64", "f32"])
        c["part"] = rng.choice(["block", "block", "block", "strided"])
        return c
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 48), n_lo=1000, n_hi=int(_log(rng, 5000, 100_000)), mix=rng.randint(1, 10**6), prec=rng.choice(["f64", "f64", "f32"]))
    if kind == "cg":
        mat = rng.choice(["p2d", "p3d"])
        side = int(_log(rng, 32, 160)) if mat == "p2d" else int(_log(rng, 10, 63))
        n_p = max(1, round(side ** (2 if mat == "p2d" else 3) / 2048))
        return dict(kind=kind, mat=mat, side=side, n_p=n_p, ppn=16, refine=rng.random() < 0.7)
    if kind == "cgstep":
        if rng.random() < 0.5:
            n = int(_log(rng, 150_000, 1_690_000))
            return dict(kind=kind, count=1, n_lo=n, n_hi=n, mix=rng.choice([-2, -3]), iters=64, prec="f32")
        return dict(kind=kind, count=rng.randint(2, 32), n_lo=1000, n_hi=int(_log(rng, 5000, 100_000)), mix=rng.randint(1, 10**6), iters=8, prec="f32")
    mat = rng.choice(["p2d", "p3d", "banded"])
    c = dict(kind=kind, mat=mat, prec=rng.choice(["f64", "f32"]))
    if mat == "banded":
        c["n"] = int(_log(rng, 10_000, 300_000))
        c["n_p"], c["ppn"] = _partition(rng, c["n"], 700, 1500)
    else:
        c["side"] = int(_log(rng, 64, 1000)) if mat == "p2d" else int(_log(rng, 16, 100))
        n = c["side"] ** (2 if mat == "p2d" else 3)
        c["n_p"], c["ppn"] = _partition(rng, n, 512, 2048)
    return c


def _small(case):
    """The matrices of a server step: (mat, side) pairs, N log-uniform in [n_lo, n_hi]; mix -2 / -3: one 2D / 3D."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        n = _log(rng, case["n_lo"], case["n_hi"])
        dim = -case["mix"] if case["mix"] < 0 else rng.choice([2, 3])
        out.append(("p2d" if dim == 2 else "p3d", max(2, int(round(n ** (1.0 / dim))))))
    return out


# --------------------------------------------------------------- matrices

_P2D = [((0, 0), 4.0), ((0, -1), -1.0), ((0, 1), -1.0), ((-1, 0), -1.0), ((1, 0), -1.0)]
_P3D = [((0, 0, 0), 6.0)] + [(tuple(d if a == b else 0 for b in range(3)), -1.0) for a in range(3) for d in (-1, 1)]


def _stencil(shape, offsets):
    strides = [math.prod(shape[a + 1:]) for a in range(len(shape))]
    offsets = sorted(offsets, key=lambda o: sum(d * s for d, s in zip(o[0], strides)))
    n = math.prod(shape)
    ids = torch.arange(n, device=DEV)
    coords = [(ids // strides[a]) % shape[a] for a in range(len(shape))]
    cols = torch.empty((n, len(offsets)), dtype=torch.int32, device=DEV)
    mask = torch.empty((n, len(offsets)), dtype=torch.bool, device=DEV)
    for q, (delta, _) in enumerate(offsets):
        ok, lin = torch.ones(n, dtype=torch.bool, device=DEV), 0
        for a, d in enumerate(delta):
            if d:
                ok &= (coords[a] + d >= 0) & (coords[a] + d < shape[a])
            lin += d * strides[a]
        mask[:, q] = ok
        cols[:, q] = (ids + lin).to(torch.int32)
    vals = torch.tensor([v for _, v in offsets], dtype=torch.float64, device=DEV).expand(n, -1)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(mask.sum(1), 0)
    return row_ptr, cols[mask], vals[mask]


def _banded(n, gen, mean=20.0, lo=4, hi=64, band=0.005, p_band=0.8):
    w = max(1, round(band * n))
    length = torch.poisson(torch.full((n,), mean, device=DEV), generator=gen).clamp(lo, min(hi, n)).to(torch.int64)
    ids = torch.arange(n, device=DEV)
    rows = torch.repeat_interleave(ids, length - 1)

    def fill(r):
        near = torch.rand(r.numel(), generator=gen, device=DEV) < p_band
        a, b = (r - w).clamp_min(0), (r + w).clamp_max(n - 1)
        cb = a + (torch.rand(r.numel(), generator=gen, device=DEV, dtype=torch.float64) * (b - a + 1)).to(torch.int64)
        return torch.where(near, cb, torch.randint(0, n, (r.numel(),), generator=gen, device=DEV))

    key = rows * n + fill(rows)
    while True:  # repeats in a row and the diagonal are drawn again
        key = torch.sort(key)[0]
        rows = torch.div(key, n, rounding_mode="floor")
        bad = key == rows * (n + 1)
        bad[1:] |= key[1:] == key[:-1]
        if not bool(bad.any()):
            break
        r = rows[bad]
        key[bad] = r * n + fill(r)
    off_val = torch.randn(key.numel(), generator=gen, device=DEV, dtype=torch.float64)
    diag = 1.0 + torch.segment_reduce(off_val.abs(), "sum", lengths=length - 1, axis=0)
    key = torch.cat([key, ids * (n + 1)])
    val = torch.cat([off_val, diag])
    key, order = torch.sort(key)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(length, 0)
    return row_ptr, (key % n).to(torch.int32), val[order]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _matrix(case, seed):
    mat = case["mat"]
    if mat == "p2d":
        return _stencil((case["side"],) * 2, _P2D)
    if mat == "p3d":
        return _stencil((case["side"],) * 3, _P3D)
    if mat == "q1":
        q1 = inputs.q1_aniso_stencil(0.001, math.pi / 8)
        return _stencil((case["side"],) * 2, [((dy, dx), v) for (dx, dy), v in q1.items()])
    return _banded(case["n"], _gen(seed + 1_000_003))


def _vector(n, seed):
    return torch.rand(n, generator=_gen(seed), device=DEV, dtype=torch.float64) * 2.0 - 1.0


def _plan(csr, n_p, ppn, prec, part="block"):
    flags = (nap.F32_VALUES if prec == "f32" else 0) | (nap.PARTITION_STRIDED if part == "strided" else 0)
    return nap.napspmv_plan(*csr, n_p, ppn, flags)


# ---------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "apply":
        csr = _matrix(case, seed)
        st["plan"] = _plan(csr, case["n_p"], case["ppn"], case["prec"], case["part"])
        st["v"] = _vector(csr[0].numel() - 1, seed)
        st["w"] = torch.empty_like(st["v"])
        st["opts"] = nap.make_opts(precision=nap.PREC_F32) if case["prec"] == "f32" else None
    elif kind == "batch":
        st["plans"], st["v"], st["w"] = [], [], []
        for q, (mat, side) in enumerate(_small(case)):
            csr = _matrix(dict(mat=mat, side=side), seed)
            n = csr[0].numel() - 1
            st["plans"].append(_plan(csr, max(1, round(n / 2048)), 16, case["prec"]))
            st["v"].append(_vector(n, seed * 1000 + q))
            st["w"].append(torch.empty_like(st["v"][-1]))
        st["opts"] = nap.make_opts(precision=nap.PREC_F32 if case["prec"] == "f32" else nap.PREC_F64)
    elif kind == "cg":
        csr = _matrix(case, seed)
        st["plan"] = _plan(csr, case["n_p"], case["ppn"], "f32")
        st["b"] = _vector(csr[0].numel() - 1, seed)
        st["x"] = torch.empty_like(st["b"])
    elif kind == "cgstep":
        mats = [(side ** (2 if mat == "p2d" else 3), mat, side) for mat, side in _small(case)]
        total = sum(n for n, _, _ in mats)
        st["x"], st["r"], p, q = torch.zeros(4, total, dtype=torch.float64, device=DEV).unbind(0)
        st["scal"] = torch.zeros(len(mats), 8, dtype=torch.float64, device=DEV)
        st["slots"], at = [], 0
        for i, (n, mat, side) in enumerate(mats):
            csr = _matrix(dict(mat=mat, side=side), seed)
            cut = slice(at, at + n)
            st["slots"].append(dict(plan=_plan(csr, max(1, round(n / 2048)), 16, case["prec"]), ws=None, b=_vector(n, seed * 1000 + i),
                                    x=st["x"][cut], r=st["r"][cut], p=p[cut], q=q[cut], scal=st["scal"][i]))
            at += n
    else:
        st["csr"] = _matrix(case, seed)
        st["v"] = _vector(st["csr"][0].numel() - 1, seed)
        st["w"] = torch.empty_like(st["v"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        if st["opts"] is not None:
            nap.napspmv_apply_ex(st["plan"], st["v"], st["w"], case["reps"], case["scale"], st["opts"])
        elif case["reps"] > 1 or case["scale"] != 1.0:
            nap.napspmv_apply_n(st["plan"], st["v"], st["w"], case["reps"], case["scale"])
        else:
            nap.napspmv_apply(st["plan"], st["v"], st["w"])
        return st["w"]
    if kind == "batch":
        nap.napspmv_apply_batch(st["plans"], st["v"], st["w"], [1] * len(st["plans"]), opts=st["opts"])
        return st["w"]
    if kind == "cg":
        st["x"].zero_()
        solve = nap.napspmv_cg_ir if case["refine"] else nap.napspmv_cg
        info = solve(st["plan"], st["b"], st["x"], rtol=1e-10)
        return dict(x=st["x"], converged=bool(info["converged"]))
    if kind == "cgstep":
        prec = nap.PREC_F32 if case["prec"] == "f32" else nap.PREC_F64
        nap.napspmv_cg_batch_init(st["slots"], prec, x_is_zero=True)
        nap.napspmv_cg_batch_iterate(st["slots"], prec, case["iters"])
        return dict(x=st["x"], r=st["r"], scal=st["scal"])
    plan = _plan(st["csr"], case["n_p"], case["ppn"], case["prec"])
    nap.napspmv_apply(plan, st["v"], st["w"])
    stats = nap.napspmv_plan_stats(plan)
    return dict(w=st["w"], stats=np.array([v for k, v in sorted(stats.items()) if isinstance(v, int)], np.int64))


# ------------------------------------------------------------------- work

def _size(case):
    """Rows and stored entries of a case's matrix."""
    if case["mat"] == "banded":
        return case["n"], 20 * case["n"]
    s = case["side"]
    return {"p2d": (s * s, 5 * s * s - 4 * s), "p3d": (s**3, 7 * s**3 - 6 * s * s), "q1": (s * s, (3 * s - 2) ** 2)}[case["mat"]]


def _product(n, nnz, prec):
    """Bytes of w <- A v: row pointer, columns and values, v, w."""
    return 4 * (n + 1) + nnz * (8 if prec == "f32" else 12) + 16 * n


def work(case):
    kind = case["kind"]
    if kind == "apply":
        n, nnz = _size(case)
        return {"bytes": case["reps"] * _product(n, nnz, case["prec"]), "flops": case["reps"] * 2 * nnz}
    if kind == "plan":
        n, nnz = _size(case)
        # the CSR once in and once laid out, and the first product
        return {"bytes": 2 * (8 * (n + 1) + 12 * nnz) + _product(n, nnz, "f64"), "flops": 2 * nnz}
    if kind == "cg":
        n, nnz = _size(case)
        # iterations to 1e-10 grow with the side; a CG iteration reads A, p, q, r, x and writes p, q, r, x
        its = (3 if case["mat"] == "p2d" else 4) * case["side"]
        return {"bytes": its * (_product(n, nnz, "f32" if case["refine"] else "f64") + 64 * n), "flops": its * (2 * nnz + 10 * n)}
    sizes = [_size(dict(mat=mat, side=side)) for mat, side in _small(case)]
    if kind == "batch":
        return {"bytes": sum(_product(n, nnz, case["prec"]) for n, nnz in sizes), "flops": sum(2 * nnz for _, nnz in sizes)}
    its = case["iters"]
    return {"bytes": sum(its * (_product(n, nnz, case["prec"]) + 64 * n) for n, nnz in sizes), "flops": sum(its * (2 * nnz + 10 * n) for n, nnz in sizes)}


# ------------------------------------------------------------------ exact

class _Csr:
    """A x in 64 bits with torch's own operations."""

    def __init__(self, csr):
        row_ptr, col, val = csr
        self.a = torch.sparse_csr_tensor(row_ptr, col.to(torch.int64), val, (row_ptr.numel() - 1,) * 2)

    def __call__(self, x):
        return torch.mv(self.a, x)


def _sine(side):
    """The orthogonal eigenvectors and the eigenvalues of the 1D second-difference matrix."""
    k = torch.arange(1, side + 1, dtype=torch.float64, device=DEV)
    s = torch.sin(math.pi / (side + 1) * k[:, None] * k[None, :]) * math.sqrt(2.0 / (side + 1))
    return s, 2.0 - 2.0 * torch.cos(math.pi / (side + 1) * k)


def _poisson_solve(b, side, dim):
    s, lam = _sine(side)
    x = b.reshape((side,) * dim)

    def transform(y):
        for a in range(dim):
            y = torch.movedim(torch.tensordot(s, y, dims=([1], [a])), 0, a)
        return y

    total = sum(lam.reshape([-1 if a == c else 1 for c in range(dim)]) for a in range(dim))
    return transform(transform(x) / total).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        a, x = _Csr(_matrix(case, seed)), None
        x = _vector(a.a.shape[0], seed)
        for _ in range(case["reps"]):
            x = case["scale"] * a(x)
        return x
    if kind == "batch":
        out = []
        for q, (mat, side) in enumerate(_small(case)):
            a = _Csr(_matrix(dict(mat=mat, side=side), seed))
            out.append(a(_vector(a.a.shape[0], seed * 1000 + q)))
        return out
    if kind == "cg":
        dim = 2 if case["mat"] == "p2d" else 3
        return dict(x=_poisson_solve(_vector(case["side"] ** dim, seed), case["side"], dim), converged=None)
    if kind == "cgstep":
        xs, rs, scal = [], [], []
        for i, (mat, side) in enumerate(_small(case)):
            a = _Csr(_matrix(dict(mat=mat, side=side), seed))
            b = _vector(a.a.shape[0], seed * 1000 + i)
            x, r, p, rr = torch.zeros_like(b), b.clone(), b.clone(), torch.dot(b, b)
            bb = rr
            for _ in range(case["iters"]):
                q = a(p)
                pq = torch.dot(p, q)
                alpha = rr / pq
                x, r = x + alpha * p, r - alpha * q
                new = torch.dot(r, r)
                beta, rr = new / rr, new
                p = r + beta * p
            xs.append(x)
            rs.append(r)
            zero = torch.zeros_like(rr)
            scal.append(torch.stack([rr, pq, alpha, beta, rr, bb, zero, zero]))
        return dict(x=torch.cat(xs), r=torch.cat(rs), scal=torch.stack(scal))
    a = _Csr(_matrix(case, seed))
    return dict(w=a(_vector(a.a.shape[0], seed)), stats=None)
