"""The allocation-free counts with a maximum range far beyond the rays, and
with rays of more pieces than the launch has rows of blocks."""
import numpy as np
import pytest
import torch

from paper_2206_06079_gb300 import ohm, synth, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _grid(max_range, corner, dims, **kw):
    return dict(dict(voxel_size=0.1, map_origin=(0.0, 0.0, 0.0), frac_bits=8, segment_steps=1 << 20, max_range=max_range,
                     corner=corner, dims=dims), **kw)


def _counts(grid, o, e, f):
    n = int(np.prod(grid["dims"]))
    hits, misses = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    ohm.count_rays_noalloc(grid, o, e, f, hits, misses)
    return hits, misses


def test_short_rays_cost_the_same_at_any_maximum_range():
    r = synth.room_scan(n=1000)
    args = r.origins.cuda(), r.endpoints.cuda(), r.flags.cuda()
    near, far = (_grid(m, (-56, -48, -5), (112, 96, 56)) for m in (12.0, 1e5))
    for x, y in zip(_counts(near, *args), _counts(far, *args)):
        assert torch.equal(x, y) and int(x.sum()) > 0
    hits, misses = (torch.zeros(112 * 96 * 56, dtype=torch.int32, device="cuda") for _ in range(2))

    def us(grid):
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                ohm.count_rays_noalloc(grid, *args, hits, misses)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 100)
        return sorted(times)[3]
    near_us, far_us = us(near), us(far)
    assert far_us < 3 * near_us, (near_us, far_us)  # 25 times, with a thread for every piece of the range


@pytest.mark.parametrize("n", [32768, 32737])
def test_rays_longer_than_the_rows_of_blocks(n):
    """Rays of up to 45 m: 38 pieces, over 20 rows for this many rays."""
    rng = np.random.default_rng(6)
    o = torch.tensor([[0.03, -0.02, 0.04]]).cuda()
    e = torch.from_numpy((rng.uniform(-1, 1, size=(n, 3)) * [45.0, 3.0, 2.0]).astype(np.float32)).cuda()
    f = torch.from_numpy((rng.random(n) < 0.3).astype(np.uint8)).cuda()
    corner, dims = (-460, -32, -22), (920, 64, 44)
    hits, misses = _counts(_grid(50.0, corner, dims, frac_bits=16), o, e, f)
    z, y, x = torch.meshgrid(*(torch.arange(d) for d in dims[::-1]), indexing="ij")
    pts = ((torch.stack([x, y, z], -1).reshape(-1, 3).double() + torch.tensor(corner).double() + 0.5) * 0.1).float().cuda()
    with ohm.Map(**W.room_params(layers=W.COUNTS, max_rays=n, max_range=50.0)) as m:
        m.integrate(o, e, f)
        want = m.query(pts, counts=True)["counts"]
    assert torch.equal(hits, want[:, 0]) and torch.equal(misses, want[:, 1])
    assert int(hits.sum()) == int((f == 0).sum())
