"""What a map reports after calls that a graph replayed: the host made no call
for them, so it has to come from the device."""
import numpy as np
import pytest
import torch

from paper_2206_06079_gb300 import ohm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _rays(n, centre):
    rng = np.random.default_rng(n)
    e = (rng.uniform(-1.0, 1.0, size=(n, 3)) + centre).astype(np.float32)
    return torch.tensor([[0.1, 0.1, 0.1]]).cuda(), torch.from_numpy(e).cuda()


def _map():
    return ohm.Map(**W.tunnel_params(max_rays=1024, max_regions=256, max_ndt_regions=64))


def test_sync_reports_a_failure_of_a_replayed_backward():
    """The NDT adjoint of rays that were never integrated finds no samples."""
    P = np.eye(3, 4)
    with _map() as m:
        o, e = _rays(256, [1.6, 1.6, 1.6])
        _, other = _rays(256, [8.0, 8.0, 8.0])
        w = torch.ones((256, 3), device="cuda"), torch.ones((256, 6), device="cuda")
        m.integrate(o, e)
        m.ndt_backward(P, o, other, None, e, *w)
        with pytest.raises(ohm.OhmError):
            m.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            m.ndt_backward(P, o, other, None, e, *w)
        m.integrate(o, e)
        m.sync()
        g.replay()
        with pytest.raises(ohm.OhmError):
            m.sync()
        m.sync()  # reported once
        m.integrate(o, e)



def test_stats_of_a_replayed_call():
    with _map() as m:
        o, e = _rays(500, [1.6, 1.6, 1.6])
        m.integrate(o, e)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            m.integrate(o, e, sync=False)
        few = e[:100].contiguous()
        m.integrate(o, few)
        assert m.stats()["rays"] == 100
        g.replay()
        s = m.stats()
        assert s["rays"] == 500 and s["visits"] > 500
        batch = ohm.Batch([m])
        batch.integrate([(o, few, None)], graph=False)
        batch.sync()
        assert m.stats()["rays"] == 100
        batch.close()
