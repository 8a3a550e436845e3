"""The batches' persistent active-node kernel at every axis length it has an
instance for: one batch of all of them, each instance against the oracle."""
import pytest

from paper_1005_5405_gb300 import binding, workloads
from tests.gpu_helpers import f_metric, make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [(12, 16, 20, 24, 28, 32), (32, 12), (28, 24, 28)])
def test_batch_of_all_lengths(lengths, monkeypatch):
    for k in ("BZ_LAZY_ORDER", "BZ_LAZY_MCAP", "BZ_LAZY_ST", "BZ_LAZY_G", "BZ_BATCH_LZ_AHEAD"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("BZ_BATCH_MODE", "lz")
    ps = [workloads.small(nx=5, ny=3, nv=nv, vmax=4.0, nt=nv * nv, seed=nv + i, lid_u0=0.1, instance=i)
          for i, nv in enumerate(lengths)]
    b = binding.Batch(ps)
    assert b.schedule()["fanout_branches"] == -1
    ref = [make(p)[1:] for p in ps]
    for i, (_, h0) in enumerate(ref):
        b.set_state(i, h0.astype("float32"), step=0)
    b.step(2)
    for i, (o, h) in enumerate(ref):
        for n in range(2):
            h, _ = o.step(h, n)
        assert f_metric(o, b.get_state(i)[0].cpu().numpy(), h) <= 2e-5   # 1e-5 a step, as in the parity tests
