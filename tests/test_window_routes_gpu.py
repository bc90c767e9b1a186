"""Which path a call takes around the staged windows, and that it answers the same on every
path: batches of plans with different default options, default options read and written back,
workspaces in error, steps and applies that a caller captured, the largest plan on windows."""
import numpy as np
import pytest
import torch

from gpu_util import gpu_plan
from paper_1612_08060_gb300 import inputs as I
from paper_1612_08060_gb300 import napspmv as nap
from test_windows_gpu import near_and_far

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


@pytest.mark.parametrize("message_less", [False, True])
def test_workspace_in_error_leaves_the_rest_of_a_windowed_batch_alone(message_less):
    """A workspace whose flag is set skips its part of the shared launches; a healthy entry,
    with messages or without, reads the vector that the launch before them wrote."""
    A, B = gpu_plan(I.poisson3d(16), 16, 4), gpu_plan(I.poisson2d(60), 1 if message_less else 20, 4)
    va, vb = vec(A.n, 1), vec(B.n, 2)
    wa, wb, vb2 = torch.full_like(va, 7.0), torch.empty_like(vb), torch.empty_like(vb)
    nap.napspmv_apply_ex(A, va, wa, 1, 1.0, nap.make_opts(engine=nap.ENGINE_FUSED, debug_stall=1, timeout_ms=50))
    torch.cuda.synchronize()
    wa.fill_(7.0)
    want = torch.empty_like(vb)
    nap.napspmv_apply_ex(B, vb, vb2, 1, 1.0, nap.make_opts(engine=nap.ENGINE_FUSED))
    nap.napspmv_apply_ex(B, vb2, want, 1, 1.0, nap.make_opts(engine=nap.ENGINE_FUSED))
    for _ in range(20):
        vb2.fill_(float("nan"))
        nap.napspmv_apply(B, vb, vb2)  # its windows end in the launch that the batch depends on
        nap.napspmv_apply_batch([A, B], [va, vb2], [wa, wb], [1, 1])
        assert torch.equal(wb, want)
    assert nap.napspmv_status(B) == nap.OK
    assert torch.all(wa == 7.0) and nap.napspmv_status(A) == nap.ERR_TIMEOUT
    nap.napspmv_apply_batch([A, B], [va, vb2], [wa, wb], [1, 1])
    assert nap.napspmv_status(A) == nap.OK and not torch.any(wa == 7.0)


TILES = dict(engine=nap.ENGINE_PHASED, pipeline=nap.PIPELINE_CTA, vec=1)
FUSED = dict(engine=nap.ENGINE_FUSED)


def short_or_long(mat):
    """A plan of short rows (without inter-node messages; without any), or of long rows whose
    far messages the windows reorder."""
    if mat != "long":
        return gpu_plan(I.poisson3d(18), *{"short": (7, 3), "one node": (7, 7), "one process": (1, 1)}[mat])
    return gpu_plan(near_and_far(300 * 80 + 1, 700, 1, 300), 80, 1)


class Steps:
    """Applies on one path or another, and the step that follows, of one plan."""

    def __init__(self, mat, prec):
        self.plan, self.prec = short_or_long(mat), prec
        self.v, self.w, self.z = vec(self.plan.n, 1), vec(self.plan.n, 2), vec(self.plan.n, 3)
        self.ws = nap.Workspace(self.plan)  # for what is expected

    def apply(self, x, path, ws=None):
        nap.napspmv_apply_ex(self.plan, x, self.w, 1, 1.0, nap.make_opts(precision=self.prec, **path), ws=ws)

    def step(self, path, ws=None):
        self.z.fill_(float("nan"))
        nap.napspmv_spmv_step(self.plan, self.v, self.z, 1.0, nap.make_opts(precision=self.prec, **path), ws=ws)
        return self.z

    def want(self, x):
        self.apply(x, TILES, self.ws)
        return bits(self.step(TILES, self.ws))


def paths(prec):  # (the fused engine leaves FP64 receives, which an FP32 step refuses)
    return [{}, TILES] if prec else [{}, TILES, FUSED]


@pytest.mark.parametrize("prec", [nap.PREC_F64, nap.PREC_F32])
@pytest.mark.parametrize("mat", ["short", "long", "one node", "one process"])
def test_captured_step_takes_the_receives_of_the_apply_before_the_replay(mat, prec):
    S = Steps(mat, prec)
    x = [vec(S.plan.n, 30 + k) for k in range(2)]
    want = [S.want(y) for y in x]
    for step in ({}, TILES):
        for before in paths(prec):
            S.ws2 = nap.Workspace(S.plan)  # nothing on it was captured yet
            S.apply(x[0], before, S.ws2)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                S.step(step, S.ws2)
            graph.replay()
            assert np.array_equal(bits(S.z), want[0]), (step, before)
            for after in paths(prec):
                S.apply(x[1], after, S.ws2)
                for _ in range(2):
                    graph.replay()
                    assert np.array_equal(bits(S.z), want[1]), (step, before, after)
                assert np.array_equal(bits(S.step({}, S.ws2)), want[1]), (step, before, after)
            del graph


@pytest.mark.parametrize("prec", [nap.PREC_F64, nap.PREC_F32])
@pytest.mark.parametrize("mat", ["short", "long", "one node", "one process"])
def test_step_after_a_capture_that_did_not_run(mat, prec):
    """An apply that was captured and not replayed changes no receives, whatever ran before."""
    S = Steps(mat, prec)
    x = [vec(S.plan.n, 40 + k) for k in range(3)]
    want = [S.want(y) for y in x]
    for one in paths(prec):
        for two in paths(prec):
            ws = nap.Workspace(S.plan)
            S.apply(x[0], one, ws)
            S.apply(x[1], two, ws)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                S.apply(x[2], {}, ws)
            assert np.array_equal(bits(S.step({}, ws)), want[1]), (one, two)
            graph.replay()
            assert np.array_equal(bits(S.step({}, ws)), want[2]), (one, two)
            S.apply(x[0], two, ws)
            assert np.array_equal(bits(S.step(TILES, ws)), want[0]), (one, two)
            del graph


def launches(plan, v, w):
    before = nap.napspmv_launch_count()
    nap.napspmv_apply(plan, v, w)
    return nap.napspmv_launch_count() - before


@pytest.mark.parametrize("mat", ["short", "long"])
def test_default_options_read_and_written_back_change_no_path(mat):
    plan = short_or_long(mat)
    v, w = vec(plan.n, 1), vec(plan.n, 2)
    assert launches(plan, v, w) == 2  # messages, windows
    d = nap.napspmv_get_default_opts(plan)
    d.timeout_ms = 700
    nap.napspmv_set_default_opts(plan, d)
    assert launches(plan, v, w) == 2
    # another tile shape is a path of its own, and stays one when written back
    nap.napspmv_set_default_opts(plan, nap.make_opts(engine=nap.ENGINE_OVERLAP, pipeline=nap.PIPELINE_CTA))
    assert launches(plan, v, w) > 2
    nap.napspmv_set_default_opts(plan, nap.napspmv_get_default_opts(plan))
    assert launches(plan, v, w) > 2
    nap.napspmv_set_default_opts(plan, nap.make_opts(engine=nap.ENGINE_PHASED, pipeline=nap.PIPELINE_SELL))
    assert launches(plan, v, w) == 2


@pytest.mark.parametrize("rows,windows", [(819199, True), (819200, False)])
def test_largest_process_on_windows(rows, windows):
    """A process's rows and receives (one here) number 819,200 at most."""
    n = 2 * rows
    cols = np.arange(n)[:, None] + np.array([-1, 0, 1])
    ok = (cols >= 0) & (cols < n)
    row_ptr = np.concatenate([[0], np.cumsum(ok.sum(1))])
    plan = gpu_plan(I.CSR(row_ptr, cols[ok].astype(np.int32), np.linspace(-1, 1, 3 * n)[:ok.sum()]), 2, 1)
    v, w, z = vec(n, 1), vec(n, 2), vec(n, 3)
    assert (launches(plan, v, w) == 2) == windows
    nap.napspmv_apply_ex(plan, v, z, 1, 1.0, nap.make_opts(**TILES))
    assert np.array_equal(bits(w), bits(z))


def test_repeated_steps_of_long_rows():
    """From some millions of entries on, the second step after an apply fills the receive
    buffers, and later ones sum from there."""
    plan = gpu_plan(near_and_far(350 * 1000 + 1, 900, 4, 3), 350, 16)
    v, w, z = vec(plan.n, 1), vec(plan.n, 2), vec(plan.n, 3)
    ws = nap.Workspace(plan)
    for prec in (nap.PREC_F64, nap.PREC_F32):
        def step(path, ws=None):
            z.fill_(float("nan"))
            before = nap.napspmv_launch_count()
            nap.napspmv_spmv_step(plan, v, z, 1.0, nap.make_opts(precision=prec, **path), ws=ws)
            return bits(z), nap.napspmv_launch_count() - before

        for seed, reps in ((5, 1), (6, 1), (7, 3)):
            x = vec(plan.n, seed)
            nap.napspmv_apply_ex(plan, x, w, reps, 0.5, nap.make_opts(precision=prec, **TILES), ws=ws)
            want = step(TILES, ws)[0]
            nap.napspmv_apply_ex(plan, x, w, reps, 0.5, nap.make_opts(precision=prec))
            counts = []
            for _ in range(4):
                got, n = step({})
                assert np.array_equal(got, want), (prec, seed)
                counts.append(n)
            # (an FP32 step converts v first)
            assert counts == ([1, 2, 1, 1] if prec == nap.PREC_F64 else [2, 3, 2, 2])
            assert np.array_equal(step(TILES)[0], want)
    assert nap.napspmv_status(plan) == 0
