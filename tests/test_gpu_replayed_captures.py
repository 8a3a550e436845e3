"""Steps that a caller captures into a CUDA graph and replays: the replays move
the step counter on the device only.  Steps, read-outs and counters that follow
on the handle must be those of the step the device has reached (against the
oracle from the handle's own state), whatever the handle's kernel, and a
capture that is never replayed must leave the handle as it was."""
import numpy as np
import pytest
import torch

from paper_1005_5405_gb300 import binding, workloads
from tests.gpu_helpers import f_metric, make, state

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-10, "f32": 1e-5}           # the per-step bounds of the parity tests


def _captured_pair(cav):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        cav.step(1)
        cav.step(1)
    return g


def _problem(nv, dtype, per_cell=False):
    return workloads.small(nx=3, ny=3, nv=nv, vmax=3.5, nt=nv * nv, seed=nv, dtype=dtype, lid_u0=0.1, kn=2.0,
                           per_cell=per_cell)


CASES = [(8, "f64", False), (15, "f32", False), (14, "f32", False), (16, "f32", False), (12, "f32", True)]


@pytest.mark.parametrize("before", [0, 5])   # steps on the handle before the capture
@pytest.mark.parametrize("nv,dtype,per_cell", CASES)
def test_steps_after_replays(nv, dtype, per_cell, before, monkeypatch):
    monkeypatch.delenv("BZ_KERNEL", raising=False)
    cav, o, _ = make(_problem(nv, dtype, per_cell))
    cav.step(before)
    g = _captured_pair(cav)
    n = before
    for replays, steps in ((20, 1), (3, 2), (1, 5)):
        for _ in range(replays):
            g.replay()
        n += 2 * replays
        torch.cuda.synchronize()
        h = state(cav)
        # An odd number of steps leaves the other buffer current: one more
        # step brings back that of the capture.
        done = 0
        for more in (steps, steps % 2):
            cav.step(more)
            for _ in range(more):
                h, mom = o.step(h, n)
                n += 1
            done += more
            assert f_metric(o, state(cav), h) <= done * TOL[dtype]
            got = cav.moments().cpu().numpy()
            assert np.max(np.abs(got - mom)) <= 10 * done * TOL[dtype] * np.max(np.abs(mom))


@pytest.mark.parametrize("nv,dtype,per_cell", CASES)
def test_counter_and_host_reads_between_replays(nv, dtype, per_cell, monkeypatch):
    """A read into host memory corrects the state in place; the next replay's
    result must again be read with its pending corrections."""
    monkeypatch.delenv("BZ_KERNEL", raising=False)
    p = _problem(nv, dtype, per_cell)
    cav, o, h = make(p)
    g = _captured_pair(cav)
    out = torch.empty((p.nr, p.nvt), dtype=cav.torch_dtype).pin_memory()
    at = binding.C.c_int64()
    for n in (0, 2, 4):
        g.replay()
        torch.cuda.synchronize()
        binding.check(binding.load().bz_get_state(cav.h, out.data_ptr(), binding.C.byref(at), None), "bz_get_state")
        torch.cuda.synchronize()
        for k in (n, n + 1):
            h, _ = o.step(h, k)
        assert f_metric(o, out.numpy(), h) <= (n + 2) * TOL[dtype]
        assert at.value == n + 2 and cav.stats()[0] == n + 2


@pytest.mark.parametrize("nv,dtype,per_cell", CASES)
def test_capture_without_a_replay(nv, dtype, per_cell, monkeypatch):
    monkeypatch.delenv("BZ_KERNEL", raising=False)
    cav, o, h = make(_problem(nv, dtype, per_cell))
    g = _captured_pair(cav)
    cav.step(3)
    for k in range(3):
        h, _ = o.step(h, k)
    got, at = cav.get_state()
    assert f_metric(o, got.cpu().numpy(), h) <= 3 * TOL[dtype]
    assert at == 3
    del g
