"""The active-node kernel at every axis length it takes (multiples of four
from 12 on, and N = 2 mod 4 from 14 on, whose threads take node pairs), with
256 and with 512 streaming threads (BZ_LAZY_ST forces the count where a plane
fits it), on a cell count that is no multiple of the group, against the oracle
after one FP32 step from the same input; and the fallback of a step whose
active nodes exceed the compact arrays (BZ_LAZY_MCAP)."""
import pytest

from paper_1005_5405_gb300 import workloads
from tests.gpu_helpers import f_metric, make, state

pytestmark = pytest.mark.gpu

SWITCHES = ("BZ_KERNEL", "BZ_LAZY_MCAP", "BZ_LAZY_G", "BZ_LAZY_TMA", "BZ_LAZY_ST", "BZ_LAZY_AHEAD")
TOL = 1e-5                                  # the FP32 step bound of the parity tests


def _problem(nv, stretched):
    grid = dict(rv=0.95, rx=0.98, ry=0.97) if stretched else {}
    return workloads.small(nx=5, ny=7, nv=nv, vmax=3.5, nt=nv * nv, seed=nv, dtype="f32", lid_u0=0.1, **grid)


def _two_steps(p):
    cav, o, h0 = make(p)
    h = state(cav)
    for n in range(2):
        cav.step(1)
        ref, _ = o.step(h, n)
        h = state(cav)
        assert f_metric(o, h, ref) <= TOL
    return cav


@pytest.mark.parametrize("stretched", [False, True])
@pytest.mark.parametrize("threads", ["256", "512"])
@pytest.mark.parametrize("nv", [12, 14, 16, 18, 20, 22, 24, 26, 28, 30, 32])
def test_step_matches_oracle(nv, threads, stretched, monkeypatch):
    for k in SWITCHES:
        monkeypatch.delenv(k, raising=False)
    if threads == "512" or nv not in (26, 30):      # (planes of 26 and 30 need 512)
        monkeypatch.setenv("BZ_LAZY_ST", threads)
    cav = _two_steps(_problem(nv, stretched))
    assert cav.get_info().kernel_variant == 2


@pytest.mark.parametrize("group", ["4", "2"])
@pytest.mark.parametrize("nv", [14, 18, 30])
def test_pairs_fallback_and_group_sizes(nv, group, monkeypatch):
    """N = 2 mod 4: two cells per group, and the generic kernel when a step
    overflows the compact arrays (also the relaxation alone)."""
    for k in SWITCHES:
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("BZ_LAZY_G", group)
    _two_steps(_problem(nv, False))
    monkeypatch.setenv("BZ_LAZY_MCAP", "8")
    p = _problem(nv, True)
    cav = _two_steps(p)
    assert cav.stats()[5] == 2              # both steps overflowed
    cav, o, h0 = make(p)
    cav.step_ex(1, 2)                       # BZ_DO_COLLIDE
    ref = o.collide(h0, 0)[0]
    assert f_metric(o, state(cav), ref) <= TOL
