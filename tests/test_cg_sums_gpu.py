"""The dot products' partition at its edges: napspmv_dot and the batched CG scalars on
inputs whose products and sums are exact in FP64 (small integers times powers of two), so
that a lost, doubled or stale partial shows whatever the order.  Lengths around a group
(256), a CTA of four groups, the whole partition (1,024 groups), a batched block (1,024
values) and a shared-memory round of partials (2,048 blocks)."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from gpu_util import gpu_plan
from paper_1612_08060_gb300 import inputs as I
from paper_1612_08060_gb300 import napspmv as nap

pytestmark = pytest.mark.gpu


def vectors(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.integers(-3, 4, n) * 0.5 ** rng.integers(0, 3, n) for _ in range(2))


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1024, 1025, 4096, 262143, 262144, 262145, 600001])
def test_dot(n):
    x, y = vectors(n, n)
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    for _ in range(2):  # the ticket is back at 0
        nap.napspmv_dot(xd, yd, n, out)
    assert Fraction(out.item()) == sum(map(Fraction, (x * y).tolist()))


@pytest.mark.parametrize("n", [64, 1023, 1025, 40000, 2048 * 1024 + 5])
def test_batched_scalars(n):
    """Two slots of one call, A = I."""
    A = I.CSR(np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.ones(n))
    plan = gpu_plan(A, 1, 1)
    slots, want = [], []
    for k in range(2):
        b, _ = vectors(n, n + k)
        z = lambda: torch.zeros(n, dtype=torch.float64, device="cuda")  # noqa: E731
        slots.append(dict(plan=plan, ws=nap.Workspace(plan), b=torch.from_numpy(b).cuda(), x=z(), r=z(), p=z(), q=z(),
                          scal=torch.zeros(8, dtype=torch.float64, device="cuda")))
        want.append(float(np.sum(b * b)))
    nap.napspmv_cg_batch_init(slots, nap.PREC_F64, x_is_zero=True)
    nap.napspmv_cg_batch_iterate(slots, nap.PREC_F64, 1)  # A = I: alpha = 1, x = b, r = 0
    for s, bb in zip(slots, want):
        scal = s["scal"].cpu().numpy()
        assert scal[5] == bb and scal[1] == bb and scal[2] == 1.0 and scal[0] == 0.0
        assert torch.equal(s["x"], s["b"]) and not s["r"].any()


@pytest.mark.parametrize("prec", [nap.PREC_F64, nap.PREC_F32])
@pytest.mark.parametrize("iters", [2, 5, 8])
def test_iterations_in_one_call(prec, iters):
    """Several iterations in one call (the direction alternating with the workspace's vector
    and sent as it is formed) against one iteration a call: the same operations, the same
    bits, and the same receives for a step afterwards."""
    mats = [(I.poisson2d(70), 5, 16, 0), (I.poisson3d(12), 4, 2, 0), (I.poisson2d(40), 20, 4, nap.PARTITION_STRIDED),
            (I.poisson2d(330), 53, 16, 0)]  # the last one past NAPSPMV_SOLO_NNZ
    runs = []
    for calls in ([iters], [1] * iters):
        slots = []
        for k, (A, n_p, ppn, fl) in enumerate(mats):
            plan = gpu_plan(A, n_p, ppn, nap.F32_VALUES | fl)
            z = lambda: torch.zeros(A.n, dtype=torch.float64, device="cuda")  # noqa: E731, B023
            slots.append(dict(plan=plan, ws=nap.Workspace(plan), b=torch.from_numpy(I.vector(A.n, k)).cuda(), x=z(), r=z(),
                              p=z(), q=z(), scal=torch.zeros(8, dtype=torch.float64, device="cuda")))
        nap.napspmv_cg_batch_init(slots, prec, x_is_zero=True)
        for c in calls:
            nap.napspmv_cg_batch_iterate(slots, prec, c)
        out = [s[f].clone() for s in slots for f in ("x", "r", "p", "q", "scal")]
        for k, s in enumerate(slots):
            assert nap.napspmv_ws_status(s["ws"]) == 0
            big = mats[k][0].nnz >= nap.SOLO_NNZ
            step = torch.empty_like(s["x"])
            nap.napspmv_spmv_step(s["plan"], s["b"], step, 1.0, nap.make_opts(precision=prec if big else nap.PREC_F64), ws=s["ws"])
            out.append(step)
        runs.append([o.cpu().numpy().view(np.int64) for o in out])
    for k, (a, b) in enumerate(zip(*runs)):
        assert np.array_equal(a, b), k
