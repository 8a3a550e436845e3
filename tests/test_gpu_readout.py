"""Read-outs of states with pending corrections: the one-pass state copy and
the FP64 moments (Eqs. densita..sforzi) taken from the stored pair."""
import numpy as np
import pytest
import torch

from paper_1005_5405_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def _problem(nv, dtype="f32", nx=5, ny=3):
    return workloads.small(nx=nx, ny=ny, nv=nv, vmax=4.0, nt=1500, seed=17, dtype=dtype, eps=0.1)


def _moments64(p, h, eps):
    """Eqs. densita..sforzi in FP64, and the L1 scale of each sum."""
    a = workloads.axis_nodes(p.nv, p.vmax)
    A = 2 * p.vmax / p.nv * np.pi ** -0.5 * np.exp(-a * a)
    vx, vy, vz = (x.ravel() for x in np.meshgrid(a, a, a, indexing="ij"))
    wx, wy, wz = (x.ravel() for x in np.meshgrid(A, A, A, indexing="ij"))
    w = wx * wy * wz
    psi = np.stack([np.ones_like(vx), vx, vy, vz, vx * vx, vy * vy, vz * vz, vx * vy, vx * vz, vy * vz])
    m = (h * w) @ psi.T
    scale = (np.abs(h) * w) @ np.abs(psi).T
    rho, n = m[:, 0], 1 + eps * m[:, 0]
    u = m[:, 1:4] / n[:, None]
    th = (2 / 3 * m[:, 4:7].sum(1) - rho) / n - 2 * eps / 3 * (u * u).sum(1)
    uu = np.stack([u[:, i] * u[:, j] for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1)
    out = np.concatenate([rho[:, None], u, th[:, None], 2 * m[:, 4:] - 2 * eps * n[:, None] * uu], 1)
    return out, scale.sum(1)


@pytest.mark.parametrize("nv", [12, 16, 20, 32])
def test_state_copy_paths_agree(nv):
    """The one-pass copy (aligned device memory), the copy to an address that
    is not 16-byte aligned and the copy to the host give the same state."""
    p = _problem(nv)
    cav = binding.Cavity(p)
    cav.set_state(workloads.warm_state(p, seed=3))
    cav.step(3)
    one = cav.get_state()[0]
    buf = torch.zeros(p.nodes + 1, dtype=torch.float32, device="cuda")
    cav.get_state(out=buf[1:])
    host = np.empty((p.nr, p.nvt), dtype=np.float32)
    cav.get_state(out=host)
    torch.cuda.synchronize()
    # FP32 rounding of h_c + (1 + eps h_c) kappa, which two kernels may contract differently.
    tol = 4 * 2.0 ** -24 * float(one.abs().max())
    assert float((one.reshape(-1) - buf[1:]).abs().max()) <= tol
    assert float(np.abs(one.cpu().numpy() - host).max()) <= tol


@pytest.mark.parametrize("nv,dtype", [(5, "f64"), (9, "f64"), (16, "f64"), (10, "f32"), (12, "f32"), (16, "f32"),
                                      (20, "f32"), (32, "f32")])
@pytest.mark.parametrize("batch", [False, True])
def test_moments_of_a_stored_state(nv, dtype, batch):
    """bz_moments of a state whose moments no step left behind, against FP64
    sums of the copied state (batches: FP32, multiples of four)."""
    p = _problem(nv, dtype)
    if batch:
        if dtype == "f64" or nv % 4:
            pytest.skip("batches take FP32 states on multiples of four nodes")
        b = binding.Batch([p, _problem(nv, nx=4, ny=4)])
        for i, q in enumerate(b.problems):
            b.set_state(i, workloads.warm_state(q, seed=4 + i))
        b.tune(1)
        b.step(3)
        got, h, eps = b.moments(0), b.get_state(0)[0], p.eps
    else:
        cav = binding.Cavity(p)
        cav.set_state(workloads.warm_state(p, seed=4))
        cav.step(3)
        cav.lid_shear()                      # the step's moments are given up
        got, h, eps = cav.moments(), cav.get_state()[0], p.eps
    ref, scale = _moments64(p, h.double().cpu().numpy(), eps)
    # FP64 sums of N^3 terms; for FP32 states the corrected node values may
    # differ by an FP32 rounding between the two read-outs.
    unit = 2.0 ** -22 if dtype == "f32" else p.nvt * 2.0 ** -53
    assert np.all(np.abs(got.cpu().numpy() - ref) <= 8 * unit * scale[:, None])
