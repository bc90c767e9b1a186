"""Staged windows (the default) against the one-lane tile pass, bit for
bit: both sum each row in its stored order with one FMA per entry, and messages are
copies, so nothing may differ.  Sizes at the edges: rows per process around 32, the
blocks' 128 and 256 rows and several blocks; send groups of 128 elements that cross
messages; strided partitions (windows without runs, two threads per row); chains; vectors
8 bytes off a 16-byte boundary; infinities, NaN and signed zeros."""
import numpy as np
import pytest
import torch

from gpu_util import gpu_plan
from paper_1612_08060_gb300 import inputs as I
from paper_1612_08060_gb300 import napspmv as nap

pytestmark = pytest.mark.gpu

TILES = dict(engine=nap.ENGINE_PHASED, pipeline=nap.PIPELINE_CTA, vec=1)


def sparse(n, per_row, seed, near=0):
    """About per_row entries a row (0 to 2 per_row), anywhere or within `near` columns."""
    rng = np.random.default_rng(seed)
    cols = []
    for i in range(n):
        k = int(rng.integers(0, 2 * per_row + 1))
        lo, hi = (max(0, i - near), min(n, i + near + 1)) if near else (0, n)
        cols.append(np.sort(rng.choice(np.arange(lo, hi), min(k, hi - lo), replace=False)))
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum([len(c) for c in cols], out=row_ptr[1:])
    col = np.concatenate(cols).astype(np.int32)
    return I.CSR(row_ptr, col, rng.uniform(-1, 1, len(col)))


def both(plan, vd, reps=1, scale=0.5, prec=nap.PREC_F64):
    out = []
    for kw in ({}, TILES):
        w = torch.full_like(vd, float("nan"))
        nap.napspmv_apply_ex(plan, vd, w, reps, scale, nap.make_opts(precision=prec, **kw))
        assert nap.napspmv_status(plan) == 0
        out.append(w.cpu().numpy().view(np.int64))
    return out


CASES = [(64, 3, 1), (65, 5, 2), (129, 7, 3), (255, 6, 4), (256, 6, 2), (257, 6, 16), (700, 3, 2), (2100, 2, 1)]


@pytest.mark.parametrize("flags", [0, nap.PARTITION_STRIDED, nap.MAP_SPLIT])
@pytest.mark.parametrize("rows,n_p,ppn", CASES)
@pytest.mark.parametrize("near", [0, 40])
def test_bits(rows, n_p, ppn, flags, near):
    A = sparse(rows * n_p + (n_p > 2), 5, rows, near)
    plan = gpu_plan(A, n_p, ppn, nap.F32_VALUES | flags)
    buf = torch.from_numpy(I.vector(A.n + 1, rows)).cuda()
    before = nap.napspmv_launch_count()
    nap.napspmv_apply(plan, buf[:A.n], torch.empty_like(buf[:A.n]))
    assert nap.napspmv_launch_count() - before == 2  # messages, windows
    for vd in (buf[:A.n], buf[1:]):
        for prec in (nap.PREC_F64, nap.PREC_F32):
            for reps in (1, 2, 3):
                a, b = both(plan, vd, reps, 0.5, prec)
                assert np.array_equal(a, b), (prec, reps)


@pytest.mark.parametrize("flags", [0, nap.PARTITION_STRIDED])
@pytest.mark.parametrize("rows,n_p,ppn,near", [(64, 3, 2, 0), (65, 9, 2, 0), (130, 7, 3, 200), (513, 5, 4, 0),
                                               (1000, 41, 8, 300)])
def test_long_rows_bits(rows, n_p, ppn, near, flags):
    """Rows of about 20 entries (the last case fills 128-row blocks)."""
    A = sparse(rows * n_p + 1, 20, rows, near)
    plan = gpu_plan(A, n_p, ppn, nap.F32_VALUES | flags)
    buf = torch.from_numpy(I.vector(A.n + 1, rows)).cuda()
    for vd in (buf[:A.n], buf[1:]):
        for prec in (nap.PREC_F64, nap.PREC_F32):
            for reps in (1, 2, 3):
                a, b = both(plan, vd, reps, 0.5, prec)
                assert np.array_equal(a, b), (prec, reps)


def near_and_far(n, near, far, seed):
    """16 columns a row within `near` of the diagonal and `far` anywhere."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)[:, None]
    cols = np.concatenate([(i + rng.integers(-near, near + 1, (n, 16))) % n, rng.integers(0, n, (n, far))], 1)
    key = np.unique(i * n + cols)
    row_ptr = np.searchsorted(key, np.arange(n + 1) * n)
    return I.CSR(row_ptr.astype(np.int64), (key % n).astype(np.int32), rng.uniform(-1, 1, len(key)))


@pytest.mark.parametrize("flags", [0, nap.MAP_SPLIT])
@pytest.mark.parametrize("rows,n_p,ppn,near,far", [(1000, 30, 4, 300, 3), (257, 64, 2, 5, 1), (300, 80, 1, 700, 1)])
def test_far_columns_in_block_order(rows, n_p, ppn, near, far, flags):
    """Messages whose elements have one user each and lie 16 apart or more are sent in
    another order (no message of the first case, the far ones of the others); the other
    engines, which read the same buffer, and the step that follows either kind of apply
    do not notice."""
    A = near_and_far(rows * n_p + 1, near, far, rows)
    plan = gpu_plan(A, n_p, ppn, nap.F32_VALUES | flags)
    vd = torch.from_numpy(I.vector(A.n, rows)).cuda()
    for prec in (nap.PREC_F64, nap.PREC_F32):
        for reps in (1, 2, 3):
            a, b = both(plan, vd, reps, 0.5, prec)
            assert np.array_equal(a, b), (prec, reps)
        steps = []
        for first in ({}, TILES):
            for then in ({}, TILES):
                w, z = torch.empty_like(vd), torch.full_like(vd, float("nan"))
                nap.napspmv_apply_ex(plan, vd, w, 1, 1.0, nap.make_opts(precision=prec, **first))
                nap.napspmv_spmv_step(plan, vd, z, 1.0, nap.make_opts(precision=prec, **then))
                assert nap.napspmv_status(plan) == 0
                steps.append(z.cpu().numpy().view(np.int64))
        assert all(np.array_equal(steps[0], z) for z in steps), prec


@pytest.mark.parametrize("make,n_p,ppn", [(lambda: I.poisson2d(47), 7, 3), (lambda: I.poisson3d(17), 5, 2),
                                          (lambda: I.aniso_q1(40), 9, 4)])
@pytest.mark.parametrize("flags", [0, nap.PARTITION_STRIDED])
def test_stencils_and_special_values(make, n_p, ppn, flags):
    A = make()
    v = I.vector(A.n, 9)
    for special in ([], [np.inf, -np.inf, np.nan, -0.0, 0.0, 5e-324, 1e308, 1e-310]):
        v[3:3 + len(special)] = special
        plan = gpu_plan(A, n_p, ppn, nap.F32_VALUES | flags)
        for prec in (nap.PREC_F64, nap.PREC_F32):
            a, b = both(plan, torch.from_numpy(v).cuda(), 1, 1.0, prec)
            x, y = a.view(np.float64), b.view(np.float64)
            assert np.array_equal(np.isnan(x), np.isnan(y))
            assert np.array_equal(a[~np.isnan(x)], b[~np.isnan(y)])


@pytest.mark.parametrize("flags", [0, nap.PARTITION_STRIDED])
@pytest.mark.parametrize("prec", [nap.PREC_F64, nap.PREC_F32])
@pytest.mark.parametrize("mat", ["short", "long"])
def test_step_keeps_the_receives_of_the_last_apply(flags, prec, mat):
    """napspmv_spmv_step multiplies a new v with the receive buffers of the last apply:
    the same on the windows, and on the tiles after an apply that kept b_{nl->l} on chip
    (also when that apply was captured and replayed)."""
    A = I.poisson3d(18) if mat == "short" else sparse(1500, 20, 5)
    plan = gpu_plan(A, 7, 3, nap.F32_VALUES | flags)
    v1, v2 = (torch.from_numpy(I.vector(A.n, s)).cuda() for s in (1, 2))
    tiles = nap.make_opts(precision=prec, **TILES)
    windows = nap.make_opts(precision=prec)

    def step(opts):
        w = torch.empty_like(v1)
        nap.napspmv_spmv_step(plan, v2, w, 1.0, opts)
        assert nap.napspmv_status(plan) == 0
        return w

    w = torch.empty_like(v1)
    nap.napspmv_apply_ex(plan, v1, w, 1, 1.0, tiles)
    want = step(tiles)
    assert not torch.equal(want, w)
    assert torch.equal(step(windows), want)
    other = torch.full_like(v1, 3.0)
    nap.napspmv_apply_ex(plan, other, w, 1, 1.0, tiles)
    nap.napspmv_apply_ex(plan, v1, w, 2, 1.0, windows)
    nap.napspmv_apply_ex(plan, v1, w, 1, 1.0, windows)
    assert torch.equal(step(tiles), want) and torch.equal(step(windows), want)
    graph, x = torch.cuda.CUDAGraph(), other.clone()
    with torch.cuda.graph(graph):
        nap.napspmv_apply_ex(plan, x, w, 1, 1.0, windows)
    nap.napspmv_apply_ex(plan, other, w, 1, 1.0, tiles)
    x.copy_(v1)
    graph.replay()
    assert torch.equal(step(tiles), want) and torch.equal(step(windows), want)


@pytest.mark.parametrize("prec", [nap.PREC_F64, nap.PREC_F32])
@pytest.mark.parametrize("own_ws", [False, True])
def test_batch_bits(prec, own_ws):
    """A batch that leaves the path open (windows of several plans in shared launches, the
    fused engine for long rows and for fewer than 64 rows per process), with unequal chains,
    against each entry alone on the fused engine; and what a step finds afterwards."""
    mats = [(I.poisson2d(33), 9, 4, 0), (I.poisson3d(11), 1, 1, 0), (sparse(700, 20, 3), 5, 2, 0),
            (I.poisson2d(12), 40, 4, 0), (I.aniso_q1(25), 4, 2, nap.PARTITION_STRIDED), (I.poisson2d(70), 5, 16, 0)]
    plans = [gpu_plan(A, n_p, ppn, nap.F32_VALUES | fl) for A, n_p, ppn, fl in mats]
    vs = [torch.from_numpy(I.vector(A.n, 60 + k)).cuda() for k, (A, *_) in enumerate(mats)]
    us = [torch.from_numpy(I.vector(A.n, 90 + k)).cuda() for k, (A, *_) in enumerate(mats)]
    reps, scale = [1, 3, 2, 1, 2, 4], [0.5, 1.0, 0.25, 0.3, 1.0, 0.125]
    ws = [nap.Workspace(p) for p in plans] if own_ws else None
    results = []
    for engine in (0, nap.ENGINE_FUSED):
        outs = [torch.full_like(v, float("nan")) for v in vs]
        nap.napspmv_apply_batch(plans, vs, outs, reps, scale, opts=nap.make_opts(engine=engine, precision=prec), ws=ws)
        for k, p in enumerate(plans):
            w = ws[k] if ws else None
            assert (nap.napspmv_ws_status(w) if w else nap.napspmv_status(p)) == 0
            step = torch.empty_like(vs[k])
            nap.napspmv_spmv_step(p, us[k], step, 1.0, ws=w)  # FP64 receives after either
            with pytest.raises(nap.NapError):
                nap.napspmv_spmv_step(p, us[k], step, 1.0, nap.make_opts(precision=nap.PREC_F32), ws=w)
            outs.append(step)
        results.append([o.cpu().numpy().view(np.int64) for o in outs])
    for a, b in zip(*results):
        assert np.array_equal(a, b)
