"""bz_info of the handles whose cells keep their increments in a slab of their
own (FP64, odd axes, per-cell sets): the launch shape of the kernel that runs,
and the steps whose plans are built together."""
import pytest
import torch

from paper_1005_5405_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def _cavity(monkeypatch, **kw):
    for k in ("BZ_KERNEL", "BZ_LAZY_AHEAD"):
        monkeypatch.delenv(k, raising=False)
    return binding.Cavity(workloads.small(nx=4, ny=4, vmax=3.5, lid_u0=0.1, **kw))


@pytest.mark.parametrize("nv,dtype,size", [(8, "f64", 8), (14, "f64", 8), (15, "f32", 4)])
def test_shared_sets(nv, dtype, size, monkeypatch):
    nt = nv * nv
    cav = _cavity(monkeypatch, nv=nv, nt=nt, dtype=dtype)
    i = cav.get_info()
    # Two slabs and the products of the set, not one slab and the products.
    assert i.kernel_variant == 0 and i.smem_bytes >= size * (2 * nv ** 3 + nt)
    assert i.threads_per_cell >= nv * nv and i.threads_per_cell % 32 == 0
    assert i.plan_batch == 32 and i.plan_end == 0
    cav.step(4)
    assert cav.get_info().plan_end == 32
    cav.step(30)
    assert cav.get_info().plan_end == 64


def test_per_cell_sets_have_no_plans(monkeypatch):
    cav = _cavity(monkeypatch, nv=16, nt=300, dtype="f32", per_cell=True)
    cav.step(2)
    i = cav.get_info()
    assert i.plan_batch == 0 and i.plan_end == 0
    assert i.smem_bytes >= 4 * 2 * 16 ** 3 and i.threads_per_cell == 512


@pytest.mark.parametrize("nv,dtype", [(8, "f64"), (16, "f32")])
def test_no_plans_ahead_after_a_capture(nv, dtype, monkeypatch):
    cav = _cavity(monkeypatch, nv=nv, nt=nv * nv, dtype=dtype)
    cav.step(2)
    assert cav.get_info().plan_batch == 32
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        cav.step(2)
    i = cav.get_info()
    assert i.plan_batch == 0 and i.plan_end == 0
