"""The phase trace of the active-node kernel (bz_phase_clocks): in an iteration
that solves the correction of the group two back, that comes first in the
collision role, before its terms, and apart from the end of streaming."""
import numpy as np
import pytest

from paper_1005_5405_gb300 import workloads
from tests.gpu_helpers import make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [16, 18, 24])           # 256 and 512 streaming threads, node pairs
def test_points_of_the_collision_role(nv, monkeypatch):
    for k in ("BZ_KERNEL", "BZ_LAZY_MCAP", "BZ_LAZY_TMA", "BZ_LAZY_ST"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("BZ_LAZY_CTAS", "1")
    cav, _, _ = make(workloads.small(nx=6, ny=4, nv=nv, vmax=4.0, nt=nv * nv, seed=nv, lid_u0=0.1))
    cav.profile(2)
    cav.step(1)
    pc = cav.phase_clocks()
    cav.profile(0)
    # Six groups of four cells: iterations 2 to 5 stream, collide and solve.
    for start, streamed, terms, sums, back, solved in pc[2:6, :6]:
        assert start < solved < terms <= sums <= back
        assert start < streamed and solved != streamed
    assert np.all(pc[2:6, :6] > 0)
