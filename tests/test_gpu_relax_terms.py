"""The sorted terms of k_relax in FP32 against the oracle where its runs and
thread counts change: fewer samples than threads, runs of one to five terms,
the samples from which a CTA gets more threads than velocity columns, several
CTAs per SM and one."""
import numpy as np
import pytest

from paper_1005_5405_gb300 import workloads
from tests.gpu_helpers import f_metric, make, state

pytestmark = pytest.mark.gpu


# One FP32 step within the 1e-5 of the step parity tests, moments within ten times it.
@pytest.mark.parametrize("nv,nt", [(7, 25), (7, 85), (7, 86), (7, 400), (15, 843), (15, 844), (21, 2315), (21, 2314),
                                   (21, 9001), (31, 7447), (31, 200)])
def test_terms_match_oracle(nv, nt, monkeypatch):
    monkeypatch.delenv("BZ_KERNEL", raising=False)
    p = workloads.small(nx=3, ny=2, nv=nv, vmax=3.5, nt=nt, seed=nv + nt, dtype="f32", lid_u0=0.1)
    cav, o, h0 = make(p)
    h = state(cav)
    for n in range(2):
        cav.step(1)
        ref, mom = o.step(h, n)
        h = state(cav)
        assert f_metric(o, h, ref) <= 1e-5
        got = cav.moments().cpu().numpy()
        assert np.max(np.abs(got - mom)) <= 1e-4 * np.max(np.abs(mom))
