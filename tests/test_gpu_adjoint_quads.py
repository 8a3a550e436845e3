"""The FP32 quad kernel of the adjoint step against the oracle's FP64 adjoint
where its layout changes: one to four velocity planes per thread, one or two
CTAs per SM, sample products inside the slabs and beside them, runs of one
term and empty runs, grids one cell wide, samples far outside the box."""
import numpy as np
import pytest

import oracle
from paper_1005_5405_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    t.cuda.set_device(0)
    return t


# FP32 against FP64: every output is a sum of some hundreds of rounded terms of
# either sign; 2e-4 of the largest entry is the bound that the FP32 adjoint of
# the 12-node case has had (and the few-sample cases add fewer terms).
@pytest.mark.parametrize("nx,ny,nv,nt,vmax", [(3, 4, 12, 1728, 4.0), (3, 4, 12, 1729, 4.0), (4, 3, 16, 300, 4.0),
                                              (1, 5, 16, 4099, 4.0), (5, 1, 20, 5000, 4.5), (3, 3, 20, 1, 4.5),
                                              (3, 2, 24, 9001, 4.5), (3, 3, 12, 7, 1.0)])
def test_adjoint_quads_match_oracle(torch, nx, ny, nv, nt, vmax):
    p = workloads.small(nx=nx, ny=ny, nv=nv, vmax=vmax, nt=nt, seed=17, dtype="f32", kn=1.0, eps=0.1)
    h = workloads.warm_state(p, seed=3).astype(np.float32)
    lam = np.random.default_rng(8).standard_normal((p.nr, p.nvt)).astype(np.float32)
    o = oracle.Oracle(**p.kwargs())
    cav = binding.Cavity(p)
    for step in (0, 1):          # the second set is built ahead, on the side stream
        ref, gref = o.adjoint_step(h.astype(np.float64), lam.astype(np.float64), step=step, wD=0.5)
        g = torch.zeros(p.nx, dtype=torch.float64, device="cuda")
        out = cav.adjoint_step(step, torch.from_numpy(h).cuda(), torch.from_numpy(lam).cuda(), grad_lid=g, wD=0.5)
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()
        assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max()
        assert np.abs(g.cpu().numpy() - gref).max() <= 2e-4 * np.abs(gref).max()
