"""Which path a call takes around the staged windows, and that it answers the same on every
path: batches of plans with different default options."""
import numpy as np
import pytest
import torch

from gpu_util import gpu_plan
from paper_1612_08060_gb300 import inputs as I
from paper_1612_08060_gb300 import napspmv as nap

pytestmark = pytest.mark.gpu


def vec(n, seed):
    return torch.from_numpy(I.vector(n, seed)).cuda()


def bits(x):
    return x.cpu().numpy().view(np.int64)


@pytest.mark.parametrize("first", [0, 1])
def test_batch_keeps_each_plans_default_precision(first):
    """opts NULL: each entry runs at its own plan's default precision, and leaves its
    receives in that of its path (FP64 after a batch)."""
    mats = [(I.poisson2d(33), 9, 4), (I.poisson3d(12), 5, 2), (I.aniso_q1(24), 4, 2)]
    plans = [gpu_plan(A, n_p, ppn, nap.F32_VALUES) for A, n_p, ppn in mats]
    precs = [nap.PREC_F32 if k % 2 == first else nap.PREC_F64 for k in range(3)]
    for p, prec in zip(plans, precs):
        nap.napspmv_set_default_opts(p, nap.make_opts(precision=prec))
    vs = [vec(p.n, 10 + k) for k, p in enumerate(plans)]
    us = [vec(p.n, 20 + k) for k, p in enumerate(plans)]
    want, got = [], []
    for fused in (True, False):
        outs = [torch.full_like(v, float("nan")) for v in vs]
        if fused:
            for p, v, w, prec in zip(plans, vs, outs, precs):
                nap.napspmv_apply_ex(p, v, w, 2, 0.5, nap.make_opts(engine=nap.ENGINE_FUSED, precision=prec))
        else:
            nap.napspmv_apply_batch(plans, vs, outs, [2, 2, 2], [0.5] * 3)
        for p, u in zip(plans, us):
            outs.append(torch.empty_like(u))
            nap.napspmv_spmv_step(p, u, outs[-1], 1.0, nap.make_opts())
            assert nap.napspmv_status(p) == 0
        (want if fused else got).extend(bits(w) for w in outs)
    for k, (a, b) in enumerate(zip(got, want)):
        assert np.array_equal(a, b), k
