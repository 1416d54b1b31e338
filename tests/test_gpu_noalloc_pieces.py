"""The allocation-free counts against the oracle's walk on rays whose pieces
end at awkward places: shorter than one piece, ending on a piece boundary,
tie-heavy lattice rays, many dominant-axis pieces, rays and a sensor outside
the grid, shared and per-ray origins."""
import numpy as np
import pytest
import torch

import oracle
from paper_2206_06079_gb300 import ohm, synth

pytestmark = pytest.mark.gpu


def _want(o, e, f, grid):
    U = 1 << grid["frac_bits"]
    dims, corner = np.array(grid["dims"]), np.array(grid["corner"])
    hits = np.zeros(tuple(dims[::-1]), np.int64)
    misses = np.zeros_like(hits)
    scale = U / grid["voxel_size"]
    q = lambda x: np.rint(x.astype(np.float64) * scale).astype(np.int64)
    rmax = grid["max_range"] * scale
    for a, b, fl in zip(q(np.broadcast_to(o, e.shape)), q(e), f):
        d = (b - a).astype(np.float64)
        length = np.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
        sample = not fl & 1
        if length > rmax:
            b, sample = a + np.rint(d * (rmax / length)).astype(np.int64), False
        v = oracle.walk(a, b) - corner
        ok = ((v >= 0) & (v < dims)).all(1)
        last = np.arange(len(v)) == len(v) - 1
        h = ok & last & sample
        np.add.at(hits, tuple(v[h].T[::-1]), 1)
        m = ok & ~(last & sample)
        np.add.at(misses, tuple(v[m].T[::-1]), 1)
    return hits.reshape(-1), misses.reshape(-1)


@pytest.mark.parametrize("kind", ["fuzz", "room", "lengths", "outside"])
def test_counts_of_pieces_match_the_oracle(kind):
    grid = dict(voxel_size=0.1, map_origin=(0.0, 0.0, 0.0), frac_bits=16, segment_steps=0, max_range=9.0,
                corner=(-41, -37, -9), dims=(83, 71, 35))
    if kind == "fuzz":
        o, e, f = synth.fuzz_rays(5, 1500, extent=3.0).numpy()
    elif kind == "room":
        o, e, f = synth.room_scan(n=1777).numpy()
        f[::5] = 1
    elif kind == "lengths":  # along each axis and a diagonal, 0 to 40 voxels in steps of a voxel
        o = np.array([[0.05, -0.05, 0.05]], np.float32)
        d = np.array([[1, 0, 0], [0, -1, 0], [0, 0, 1], [0.6, -0.5, 0.2]])
        e = (o + (d[:, None] * (np.arange(41)[None, :, None] * 0.1)).reshape(-1, 3)).astype(np.float32)
        f = (np.arange(len(e)) % 3 == 0).astype(np.uint8)
    else:
        rng = np.random.default_rng(3)
        o = np.array([[60.0, 2.0, 0.0]], np.float32)
        e = (np.array([0, 0, 1.0]) + rng.uniform(-70, 70, size=(900, 3)) * [1, 0.05, 0.02]).astype(np.float32)
        f = np.zeros(900, np.uint8)
        grid.update(max_range=120.0, segment_steps=4000)
    n = grid["dims"][0] * grid["dims"][1] * grid["dims"][2]
    hits = torch.zeros(n, dtype=torch.int32, device="cuda")
    misses = torch.zeros(n, dtype=torch.int32, device="cuda")
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    ohm.count_rays_noalloc(grid, t(o), t(e), t(f), hits, misses)
    wh, wm = _want(o, e, f, grid)
    assert np.array_equal(hits.cpu().numpy(), wh)
    assert np.array_equal(misses.cpu().numpy(), wm)
    assert wm.sum() > 0
