"""Sliced rows built on the device: windows of 1, 31, 32, 33 and 1025 rows (one process
each), row lengths that are empty, equal, spread over every factor of two, at the
256-entry limit and past it, contiguous and strided.  Each row is summed in its stored
order by one lane, so the sliced pass must give the bits of the one-lane tile pass, and
both stay within 1e-13 (|A||v|)_i of the oracle (at most 300 products of one FMA each:
300 * 2^-53 = 3.4e-14)."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import abs_row_bound, assert_close_fp64, gpu_plan
from paper_1612_08060_gb300 import inputs as I
from paper_1612_08060_gb300 import napspmv as nap

pytestmark = pytest.mark.gpu


def ragged(n, kind, seed):
    rng = np.random.default_rng(seed)
    top = min(n, 300)
    if kind == "empty":
        length = np.zeros(n, np.int64)
    elif kind == "equal":
        length = np.full(n, min(top, 5))
    elif kind == "limit":
        length = rng.choice([0, 1, 2, min(top, 128), min(top, 255), min(top, 256), min(top, 257), top], n)
    else:
        length = np.minimum(top, 2 ** rng.integers(0, 9, n) - rng.integers(0, 2, n))
    cols = [np.sort(rng.choice(n, int(k), replace=False)) for k in length]
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(length, out=row_ptr[1:])
    col = np.concatenate(cols + [np.zeros(0, np.int64)]).astype(np.int32)
    return I.CSR(row_ptr, col, rng.uniform(-1, 1, len(col)))


@pytest.mark.parametrize("kind", ["empty", "equal", "limit", "spread"])
@pytest.mark.parametrize("rows,n_p,flags", [(1, 40, 0), (31, 11, 0), (32, 11, 0), (33, 11, 0), (1025, 2, 0),
                                            (33, 11, nap.PARTITION_STRIDED), (1025, 2, nap.PARTITION_STRIDED)])
def test_bits_of_the_tile_pass(kind, rows, n_p, flags):
    A = ragged(rows * n_p, kind, rows + n_p)
    v = I.vector(A.n, 3)
    plan = gpu_plan(A, n_p, 4, nap.F32_VALUES | flags)
    vd = torch.from_numpy(v).cuda()
    for prec in (nap.PREC_F64, nap.PREC_F32):
        out = []
        for pipe in (nap.PIPELINE_SELL, nap.PIPELINE_CTA):
            w = torch.full_like(vd, float("nan"))
            # a tile of its own for rows past the tile size: keep every row inside one
            o = nap.make_opts(engine=nap.ENGINE_PHASED, pipeline=pipe, precision=prec, vec=1, tile_rows=64, tile_nnz=1024)
            nap.napspmv_apply_ex(plan, vd, w, 1, 1.0, o)
            assert nap.napspmv_status(plan) == 0
            out.append(w.cpu().numpy())
        short = np.diff(A.row_ptr) <= 256  # longer rows: a warp's tree sum
        assert np.array_equal(out[0][short].view(np.int64), out[1][short].view(np.int64))
        if prec == nap.PREC_F64:
            for w in out:
                assert_close_fp64(w, O.spmv(A.row_ptr, A.col, A.val, v), abs_row_bound(A, v))


@pytest.mark.parametrize("n,n_p,ppn,flags", [(16383, 1, 1, 0), (16384, 3, 2, 0), (16385, 1, 1, 0), (32769, 2, 1, 0),
                                             (32768 + 31, 700, 3, 0), (16385, 5, 2, nap.PARTITION_STRIDED)])
@pytest.mark.parametrize("rows,nnz", [(1, 32), (33, 64), (512, 1536), (4000, 6000)])
def test_tiles_around_a_segment(n, n_p, ppn, flags, rows, nnz):
    """Row tiles are cut in segments of 16,384 rows: every row in one tile of each list,
    whatever the tile shape, so the tile passes give the sliced pass's bits."""
    rng = np.random.default_rng(n + rows)
    length = rng.integers(0, 9, n)
    length[rng.integers(0, n, 5)] = 150  # past the smaller tiles
    off = np.arange(150) * 7
    cols = [np.sort((i + off[:k]) % n) for i, k in enumerate(length)]
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(length, out=row_ptr[1:])
    A = I.CSR(row_ptr, np.concatenate(cols).astype(np.int32), rng.uniform(-1, 1, int(row_ptr[-1])))
    plan = gpu_plan(A, n_p, ppn, flags)
    vd = torch.from_numpy(I.vector(n, 2)).cuda()
    out = {}
    for engine in (nap.ENGINE_PHASED, nap.ENGINE_OVERLAP):
        for pipe in (nap.PIPELINE_SELL, nap.PIPELINE_CTA, nap.PIPELINE_WARP):
            w = torch.full_like(vd, float("nan"))
            o = nap.make_opts(engine=engine, pipeline=pipe, vec=1, tile_rows=rows, tile_nnz=nnz)
            nap.napspmv_apply_ex(plan, vd, w, 1, 1.0, o)
            assert nap.napspmv_status(plan) == 0
            out[engine, pipe] = w.cpu().numpy()
    short = length < 150  # a row past a tile is a tree sum
    want = out[nap.ENGINE_PHASED, nap.PIPELINE_SELL]
    for w in out.values():
        assert np.array_equal(w[short].view(np.int64), want[short].view(np.int64))
        assert_close_fp64(w, want, abs_row_bound(A, vd.cpu().numpy()))
