"""The cells with separate increments (FP64 states, odd velocity axes,
per-cell sets) against the oracle: one step at a time from the GPU's state,
over the edge of a batch of plans; the relaxation alone and the split step;
and steps captured by the caller, replayed past the steps of the capture."""
import numpy as np
import pytest
import torch

from paper_1005_5405_gb300 import binding, workloads
from tests.gpu_helpers import f_metric, make, state

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-10, "f32": 1e-5}           # the per-step bounds of the parity tests


def _problem(nv, dtype, per_cell=False, nt=None, nx=4, ny=3, **kw):
    return workloads.small(nx=nx, ny=ny, nv=nv, vmax=3.5, nt=nt or nv * nv, seed=nv, dtype=dtype, lid_u0=0.1,
                           per_cell=per_cell, **kw)


@pytest.mark.parametrize("nv,dtype,per_cell", [
    (5, "f64", False), (8, "f64", False), (11, "f64", False), (12, "f64", False), (14, "f64", False),
    (16, "f64", False), (18, "f64", False), (22, "f64", False), (24, "f64", False), (7, "f32", False),
    (15, "f32", False), (31, "f32", False), (9, "f64", True), (12, "f64", True), (11, "f32", True),
    (18, "f32", True), (24, "f32", True), (28, "f32", True)])
@pytest.mark.parametrize("stretched", [False, True])
def test_step_matches_oracle(nv, dtype, per_cell, stretched, monkeypatch):
    monkeypatch.delenv("BZ_KERNEL", raising=False)
    kw = dict(rx=0.98, ry=0.97) if stretched else {}
    if stretched and nv % 2 == 0:
        kw["rv"] = 0.95
    cav, o, h0 = make(_problem(nv, dtype, per_cell, **kw))
    cav.set_state(h0, step=31)              # (a batch of plans holds 32 steps at most)
    h = state(cav)
    for n in range(31, 34):
        cav.step(1)
        ref, mom = o.step(h, n)
        h = state(cav)
        assert f_metric(o, h, ref) <= TOL[dtype]
        got = cav.moments().cpu().numpy()
        assert np.max(np.abs(got - mom)) <= 10 * TOL[dtype] * np.max(np.abs(mom))


@pytest.mark.parametrize("nv,dtype,per_cell", [(12, "f64", False), (15, "f32", False), (16, "f32", True)])
def test_substeps(nv, dtype, per_cell):
    p = _problem(nv, dtype, per_cell)
    for flags in (2, 4):                    # BZ_DO_COLLIDE, BZ_SPLIT
        cav, o, h0 = make(p)
        cav.step_ex(2, flags)
        h = h0
        for n in range(2):
            h = o.collide(h, n)[0] if flags == 2 else o.step(h, n)[0]
        assert f_metric(o, state(cav), h) <= 4 * TOL[dtype]


def test_many_cells_per_cta():
    """More cells than CTAs, on more than one segment of a column or one."""
    for nx, ny in ((23, 17), (41, 37)):
        p = _problem(6, "f64", nx=nx, ny=ny, nt=300)
        cav, o, h0 = make(p)
        cav.step(1)
        assert f_metric(o, state(cav), o.step(h0, 0)[0]) <= TOL["f64"]


@pytest.mark.parametrize("nv,dtype", [(8, "f64"), (14, "f32"), (16, "f32")])
def test_captured_steps_replay_past_the_capture(nv, dtype):
    """Two steps captured by the caller and replayed 20 times are 40 steps."""
    p = _problem(nv, dtype, nx=3, ny=3, kn=2.0)
    cav, o, h0 = make(p)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        cav.step(1)
        cav.step(1)
    for _ in range(20):
        g.replay()
    torch.cuda.synchronize()
    h, _ = o.run(h0, 40)
    assert f_metric(o, state(cav), h) <= 40 * TOL[dtype]
