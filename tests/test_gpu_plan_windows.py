"""Which steps' sample plans are built ahead (bz_info.plan_end): K at a time on a
march; the K that end below a window already built on a sweep backwards in
segments; only the call's own after a jump of the step counter.  Every step
on the way against the oracle."""
import pytest

from paper_1005_5405_gb300 import binding, workloads
from tests.gpu_helpers import f_metric, make, state

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-10, "f32": 1e-5}           # the per-step bounds of the parity tests
CASES = [(8, "f64"), (15, "f32"), (14, "f32"), (16, "f32")]


def _make(nv, dtype, monkeypatch):
    for k in ("BZ_KERNEL", "BZ_LAZY_AHEAD", "BZ_LAZY_ORDER"):
        monkeypatch.delenv(k, raising=False)
    p = workloads.small(nx=3, ny=2, nv=nv, vmax=3.5, nt=nv * nv, seed=nv, dtype=dtype, lid_u0=0.1)
    cav, o, h0 = make(p)
    return cav, o, h0, TOL[dtype]


def _step_from(cav, o, h0, n, calls, tol):
    """The steps of `calls` (steps per call) from h0 at step n."""
    cav.set_state(h0, step=n)
    h = h0
    for k in calls:
        cav.step(k)
        for _ in range(k):
            h, _ = o.step(h, n)
            n += 1
    assert f_metric(o, state(cav), h) <= sum(calls) * tol
    return cav.get_info().plan_end


@pytest.mark.parametrize("nv,dtype", CASES)
def test_sweep_backwards_in_segments(nv, dtype, monkeypatch):
    cav, o, h0, tol = _make(nv, dtype, monkeypatch)
    K = cav.get_info().plan_batch
    assert K >= 2
    cav.step(2 * K)
    assert cav.get_info().plan_end == 2 * K
    ends = [_step_from(cav, o, h0, s, (1, 2), tol) for s in range(2 * K - 4, -1, -4)]
    # One batch more on the way down: the K that end where the window began.
    assert ends == [2 * K if s >= K else K for s in range(2 * K - 4, -1, -4)]


@pytest.mark.parametrize("nv,dtype", CASES)
def test_segments_across_the_edge_of_a_window(nv, dtype, monkeypatch):
    cav, o, h0, tol = _make(nv, dtype, monkeypatch)
    K = cav.get_info().plan_batch
    assert _step_from(cav, o, h0, 100, (1,), tol) == 100 + K        # a first batch
    assert _step_from(cav, o, h0, 99, (2,), tol) == 101             # [101 - K, 101)
    assert _step_from(cav, o, h0, 101 - K, (2, 1), tol) == 101
    assert _step_from(cav, o, h0, 100, (2,), tol) == 100 + K        # the march goes on
    assert _step_from(cav, o, h0, 100 + K, (3,), tol) == 100 + 2 * K
    if K < 100:
        assert _step_from(cav, o, h0, K - 5, (1,), tol) == K - 4    # (a jump)
        assert _step_from(cav, o, h0, 3, (3,), tol) == K - 5        # cut off at step 0
        assert _step_from(cav, o, h0, 0, (2, 2), tol) == K - 5


@pytest.mark.parametrize("nv,dtype", CASES)
def test_jumps(nv, dtype, monkeypatch):
    cav, o, h0, tol = _make(nv, dtype, monkeypatch)
    K = cav.get_info().plan_batch
    assert _step_from(cav, o, h0, 7, (1,), tol) == 7 + K            # a first batch
    assert _step_from(cav, o, h0, 1000, (1,), tol) == 1001          # a jump: the call's own step
    assert _step_from(cav, o, h0, 1001, (1, 1), tol) == 1001 + K    # and the march goes on
    assert _step_from(cav, o, h0, 5000, (6,), tol) == 5006
    assert _step_from(cav, o, h0, 9000, (K + 5,), tol) == 9000 + 2 * K
    assert _step_from(cav, o, h0, 20, (3,), tol) == 23
    cav.step_ex(1, 2)                                               # BZ_DO_COLLIDE
    assert cav.get_info().plan_end == 23 + K


def test_batches_jump_and_go_back(monkeypatch):
    for k in ("BZ_LAZY_AHEAD", "BZ_LAZY_ORDER", "BZ_LAZY_MCAP", "BZ_BATCH_LZ_AHEAD"):
        monkeypatch.delenv(k, raising=False)
    ps = [workloads.small(nx=3, ny=3, nv=nv, vmax=3.5, nt=400, seed=nv, lid_u0=0.1, instance=nv) for nv in (12, 16)]
    for mode in ("fanout", "lz"):
        monkeypatch.setenv("BZ_BATCH_MODE", mode)
        b = binding.Batch(ps)
        ref = [make(p)[1:] for p in ps]
        for n, k in ((3, 2), (700, 1), (701, 2), (696, 3), (2, 3)):
            for i, (o, h0) in enumerate(ref):
                b.set_state(i, h0.astype("float32"), step=n)
            b.step(k)
            for i, (o, h0) in enumerate(ref):
                h = h0
                for q in range(k):
                    h, _ = o.step(h, n + q)
                assert f_metric(o, b.get_state(i)[0].cpu().numpy(), h) <= k * TOL["f32"]
