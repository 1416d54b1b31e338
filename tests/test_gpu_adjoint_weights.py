"""The adjoints' upstream weights: queries that share voxels are summed in
double, so the gradients depend neither on the order in which the queries
arrive nor on how the sums' rows are laid out (one per query, or one per voxel
where there are more queries than voxels)."""
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


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda()


def _ndt_frame(n_query, seed=0):
    """2,048 rays whose samples lie in one region, and n_query queries in 300
    of the sample voxels, with positive weights (no cancellation in a sum)."""
    rng = np.random.default_rng(seed)
    e = rng.uniform(0.3, 2.9, size=(2048, 3)).astype(np.float32)
    q = e[rng.integers(0, 300, n_query)]
    return e, q, np.abs(rng.normal(size=(n_query, 3))) + 0.1, np.abs(rng.normal(size=(n_query, 6))) + 0.1


def _ndt_gradients(frame, order, max_ndt):
    e, q, gm, gc = frame
    P = np.eye(3, 4)
    o = _cuda([[0.15, 0.15, 0.15]])
    with ohm.Map(**W.tunnel_params(max_rays=2048, max_regions=64, max_ndt_regions=max_ndt)) as m:
        m.integrate_posed(P, o, _cuda(e))
        ge, gt = m.ndt_backward(P, o, _cuda(e), None, _cuda(q[order]), _cuda(gm[order]), _cuda(gc[order]))
        m.sync()
        return ge.cpu().numpy().astype(np.float64), gt.cpu().numpy()


@pytest.mark.parametrize("n_query", [12000, 40000])
def test_ndt_gradients_do_not_depend_on_the_order_of_queries(n_query):
    frame = _ndt_frame(n_query)
    rng = np.random.default_rng(1)
    ge, gt = _ndt_gradients(frame, np.arange(n_query), 4)  # 131,072 voxels: a row per query
    assert np.abs(gt).min() > 0
    # a sum of k positive doubles is within k 2^-53 of itself in any order: the
    # weights (at most n_query of a voxel), then the twist over the rays
    e = frame[0].astype(np.float64)
    size = np.abs(ge).sum(), (np.linalg.norm(e, axis=1) * np.linalg.norm(ge, axis=1)).sum()
    tol = np.repeat(size, 3) * (n_query + len(e)) * 2.0 ** -52
    for order, max_ndt in ((np.arange(n_query)[::-1], 4), (rng.permutation(n_query), 4), (rng.permutation(n_query), 1)):
        ge2, gt2 = _ndt_gradients(frame, order, max_ndt)  # one block, 32,768 voxels: a row per voxel of 40,000 queries
        assert (np.abs(gt2 - gt) <= tol).all(), (gt2 - gt, tol)
        # float outputs of doubles that agree to 1e-11: adjacent floats at most
        assert (np.abs(ge2 - ge) <= np.abs(ge) * 2.0 ** -23).all()


@pytest.mark.parametrize("captured, between", [(500, 30000), (30000, 500), (30000, 60000)])
def test_ndt_weights_replayed_from_a_graph(captured, between):
    """A captured backward whose queries fit the rows that the map has, and
    captured ones that do not; calls of other sizes, the map's rows growing,
    in between."""
    frame, other = _ndt_frame(captured), _ndt_frame(between, seed=3)
    P = np.eye(3, 4)
    o, e = _cuda([[0.15, 0.15, 0.15]]), _cuda(frame[0])
    a = [_cuda(x) for x in frame[1:]]
    b = [_cuda(x) for x in other[1:]]
    first = [x[:500] for x in a]
    with ohm.Map(**W.tunnel_params(max_rays=2048, max_regions=64, max_ndt_regions=4)) as m:
        m.integrate_posed(P, o, e)
        m.ndt_backward(P, o, e, None, *first)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            got = m.ndt_backward(P, o, e, None, *a)
        want_b = m.ndt_backward(P, o, e, None, *b)
        want = m.ndt_backward(P, o, e, None, *a)
        for _ in range(2):
            g.replay()
            got_b = m.ndt_backward(P, o, e, None, *b)
        torch.cuda.synchronize()
        for x, y in ((got, want), (got_b, want_b)):
            n = captured + between + len(frame[0])
            assert y[0].abs().max() > 0
            assert (x[0] - y[0]).abs().max() <= y[0].abs().max() * 2.0 ** -23
            assert (x[1] - y[1]).abs().max() <= y[1].abs().max() * n * 2.0 ** -52


@pytest.mark.parametrize("n_query", [8000, 40000])
def test_tsdf_gradients_do_not_depend_on_the_order_of_queries(n_query):
    """A 32 x 24 frame onto a wall inside one region, queries in 150 band
    voxels with positive weights."""
    rng = np.random.default_rng(2)
    w, h = 32, 24
    K, pose = (60.0, 60.0, 15.5, 11.5), np.concatenate([np.eye(3), np.full((3, 1), 0.8)], 1)
    pose[2, 3] = 0.25
    depth = _cuda(0.7 + 0.02 * rng.random((h, w)))
    vox = np.stack(np.meshgrid(np.arange(12, 20), np.arange(12, 20), np.arange(16, 22)), -1).reshape(-1, 3)[rng.permutation(384)[:150]]
    pts = (vox + 0.5)[rng.integers(0, 150, n_query)] * 0.05
    g = np.abs(rng.normal(size=n_query)) + 0.1

    def gradients(order, max_regions):
        with ohm.Map(**W.tsdf_params(max_rays=w * h, max_regions=max_regions)) as m:
            m.integrate_depth(depth, K, pose)
            assert m.region_count() == 1
            gd, gt = m.tsdf_backward(depth, K, pose, _cuda(pts[order]), _cuda(g[order]))
            m.sync()
            return gd.cpu().numpy().astype(np.float64), gt.cpu().numpy()

    gd, gt = gradients(np.arange(n_query), 2)  # 65,536 voxels: a row per query
    assert np.abs(gd).max() > 0
    for order, regions in ((np.arange(n_query)[::-1], 2), (rng.permutation(n_query), 2), (rng.permutation(n_query), 1)):
        gd2, gt2 = gradients(order, regions)  # 32,768 voxels: a row per voxel of 40,000 queries
        # each weight enters as the float nearest to its double sum, which the
        # order moves by n_query 2^-53 of itself: for 150 voxels no float changes
        assert np.array_equal(gd2, gd)
        # the pixels' float contributions (under 2 m from the origin) summed in double
        assert np.abs(gt2 - gt).max() <= 4 * np.abs(gd).sum() * gd.size * 2.0 ** -52
