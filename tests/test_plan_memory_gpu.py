"""A plan's peak memory is that of its build: the staged windows, which come last, take none
that a plan without them would not have needed."""
import pytest
import torch

from gpu_util import gpu_plan
from paper_1612_08060_gb300 import inputs as I
from paper_1612_08060_gb300 import napspmv as nap
from test_windows_gpu import near_and_far

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def plan_in(A, n_p, ppn, flags, room):
    """A plan built with `room` bytes of the device free, or None where they do not do."""
    fill = torch.empty(free() - room, dtype=torch.uint8, device="cuda")
    try:
        return gpu_plan(A, n_p, ppn, flags)
    except nap.NapError as e:
        assert e.code == nap.ERR_OOM
        return None
    finally:
        del fill
        free()


def test_windows_need_no_more_room_than_the_build():
    A, n_p, ppn = near_and_far(1000 * 1000, 900, 3, 4), 1000, 16
    w = torch.empty(A.n, dtype=torch.float64, device="cuda")
    v = torch.from_numpy(I.vector(A.n, 1)).cuda()
    for flags in (0, nap.COMPOSED_GATHERS):  # (kernels are loaded before memory is short)
        plan = gpu_plan(A, n_p, ppn, nap.F32_VALUES | flags)
        nap.napspmv_apply(plan, v, w)
        nap.napspmv_apply_ex(plan, v, w, 1, 1.0, nap.make_opts(engine=nap.ENGINE_PHASED, pipeline=nap.PIPELINE_CTA, vec=1))
        del plan
    want = w.clone()
    lo, hi = 64 * MIB, 4096 * MIB
    while hi - lo > 16 * MIB:  # the least room that does without windows
        mid = (lo + hi) // 2
        ok = plan_in(A, n_p, ppn, nap.F32_VALUES | nap.COMPOSED_GATHERS, mid) is not None
        lo, hi = (lo, mid) if ok else (mid, hi)
    plan = plan_in(A, n_p, ppn, nap.F32_VALUES, hi + 16 * MIB)
    assert plan is not None, hi // MIB
    nap.napspmv_apply(plan, v, w)
    assert nap.napspmv_status(plan) == 0
    assert torch.equal(w, want)
