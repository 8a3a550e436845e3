"""The moments of an FP32 step follow from 30 sums and the correction, not from
the stored state (the active-node kernel; odd axes and per-cell sets).  They
must be as close to those of the exact step as FP32 sums over the stored state
are."""
import numpy as np
import pytest

from paper_1005_5405_gb300 import workloads
from tests.gpu_helpers import make, state

pytestmark = pytest.mark.gpu
F = np.float32


def _sums_of_state(h, o, nv):
    """Moments from the stored FP32 states by FP32 sums: over the columns (a
    node's product and addition rounded once), then over groups of 32 columns."""
    v = o.velocities()[:nv, 2]
    j = np.arange(nv)
    a = np.cbrt(o.weights().reshape(nv, nv, nv)[j, j, j])
    x = h.astype(F).reshape(len(h), nv, nv * nv)
    y, z = np.repeat(v.astype(F), nv), np.tile(v.astype(F), nv)
    ayz = np.outer(a.astype(F), a.astype(F)).reshape(-1)
    s = []
    for k in range(3):
        t, acc = (a * v ** k).astype(F), np.zeros(x[:, 0].shape, F)
        for i in range(nv):
            acc = (t[i].astype(float) * x[:, i].astype(float) + acc).astype(F)
        s.append(acc * ayz)
    m = []
    for t in (s[0], s[1], s[0] * y, s[0] * z, s[2], s[0] * y * y, s[0] * z * z, s[1] * y, s[1] * z, s[0] * y * z):
        t = np.pad(t, ((0, 0), (0, -nv * nv % 32))).reshape(len(h), -1, 32)
        while t.shape[2] > 1:
            t = t[:, :, ::2] + t[:, :, 1::2]
        m.append(t.astype(float).sum((1, 2)))
    m, e = np.array(m), o.eps
    n = 1 + e * m[0]
    u = m[1:4] / n
    out = [m[0], *u, ((2 / 3) * m[4:7].sum(0) - m[0]) / n - (2 * e / 3) * (u * u).sum(0)]
    out += [2 * m[4 + k] - 2 * e * n * u[b] * u[c]
            for k, (b, c) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)))]
    return np.array(out).T.astype(F)


@pytest.mark.parametrize("nv,nt,per_cell", [(9, 400, False), (11, 700, False), (13, 1200, False), (15, 2500, False),
                                            (21, 4000, False), (12, 1000, True), (17, 3000, True),
                                            (14, 1500, False), (22, 4000, False), (30, 6000, False),
                                            (16, 2000, False), (24, 4000, False), (32, 6000, False)])
def test_step_moments_are_as_exact_as_sums_of_the_state(nv, nt, per_cell, monkeypatch):
    """Norms of the errors over 256 cells, eleven moments and two steps: these
    5632 errors leave about 3% of chance in either norm, so 10% between the two."""
    monkeypatch.delenv("BZ_KERNEL", raising=False)
    p = workloads.small(nx=16, ny=16, nv=nv, vmax=3.5, nt=nt, seed=nv, dtype="f32", lid_u0=0.1, per_cell=per_cell)
    cav, o, _ = make(p)
    h = state(cav)
    got, ref, exact = [], [], []
    for n in range(2):
        cav.step(1)
        exact.append(o.step(h, n)[1])
        got.append(cav.moments().cpu().numpy())
        h = state(cav)
        ref.append(_sums_of_state(h, o, nv))
    exact = np.array(exact)
    assert np.linalg.norm(np.array(got) - exact) <= 1.1 * np.linalg.norm(np.array(ref) - exact)
