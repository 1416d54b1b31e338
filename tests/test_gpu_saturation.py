"""Saturation bits of the miss walk (DeviceMap::sat): voxels driven to l_min,
lifted again by hits and passed through again must hold exactly the oracle's
log-odds, also after their regions were evicted and restored, and for clamp
bounds that are reached at once, never, or lie at the prior."""
import numpy as np
import pytest
import torch

import oracle
from paper_2206_06079_gb300 import ohm, workloads as W
from .parity import compare_dense

pytestmark = pytest.mark.gpu


def _fan(n, seed, reach):
    """n rays from one point into a narrow cone, so that they share voxels."""
    rng = np.random.default_rng(seed)
    d = np.array([1.0, 0.13, -0.07]) + 0.08 * rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    o = np.array([[0.21, -0.37, 0.11]], np.float32)
    return o, (o + reach * d).astype(np.float32)


@pytest.mark.parametrize("evict", [False, True])
@pytest.mark.parametrize("l_min", [-2.0, -0.4, 0.0, -40.0])
@pytest.mark.parametrize("layers", [W.OCC, W.OCC | W.COUNTS | W.NDT])
def test_saturated_voxels_follow_the_oracle(layers, l_min, evict):
    p = W.room_params(layers=layers | W.COUNTS, l_min=l_min, max_regions=64, max_ndt_regions=64, max_rays=4096)
    with ohm.Map(**p) as gm:
        om = oracle.OracleMap(**W.oracle_params(p))
        # misses only (no sample), then samples in the saturated cone, then misses again
        for k, (reach, flag) in enumerate([(9.0, 1), (9.0, 1), (4.0, 0), (9.0, 1), (6.0, 0), (9.0, 1)]):
            o, e = _fan(1500 + 31 * k, 7 + k, reach)
            f = np.full(len(e), flag, np.uint8)
            gm.integrate(o, e, f)
            om.integrate(o, e, f)
            if evict and k % 2 == 1:
                gm.evict(1)
                gm.restore_all()
        if not evict:
            assert compare_dense(gm, om) > 3
        pts = np.concatenate([_fan(3000, 99, r)[1] for r in (0.5, 2.0, 3.9, 4.0, 5.9, 8.0)])
        g, r = gm.query(torch.from_numpy(pts).cuda(), counts=True), om.query(pts)
        known = r["known"] == 1
        assert np.array_equal(g["known"].cpu().numpy(), r["known"]) and known.sum() > 1000
        assert np.array_equal(g["occupancy"].cpu().numpy()[known].view(np.uint32), r["occupancy"][known].view(np.uint32))
