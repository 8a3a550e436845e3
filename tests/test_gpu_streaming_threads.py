"""The active-node kernel with 256 and with 512 streaming threads against the
oracle, at every axis length it takes and a cell count that is no multiple of
the group (BZ_LAZY_ST forces the count; one FP32 step from the oracle's input)."""
import numpy as np
import pytest

from paper_1005_5405_gb300 import workloads
from tests.gpu_helpers import f_metric, make, state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretched", [False, True])
@pytest.mark.parametrize("threads", ["256", "512"])
@pytest.mark.parametrize("nv", [12, 16, 20, 24, 28, 32])
def test_step_matches_oracle(nv, threads, stretched, monkeypatch):
    for k in ("BZ_KERNEL", "BZ_LAZY_MCAP", "BZ_LAZY_G", "BZ_LAZY_TMA"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("BZ_LAZY_ST", threads)
    grid = dict(rv=0.95, rx=0.98, ry=0.97) if stretched else {}
    p = workloads.small(nx=5, ny=7, nv=nv, vmax=3.5, nt=nv * nv, seed=nv, dtype="f32", lid_u0=0.1, **grid)
    cav, o, h0 = make(p)
    assert cav.get_info().kernel_variant == 2
    h = state(cav)
    for n in range(2):
        cav.step(1)
        ref, _ = o.step(h, n)
        h = state(cav)
        assert f_metric(o, h, ref) <= 1e-5      # the FP32 step bound of the parity tests
