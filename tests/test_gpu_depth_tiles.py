"""Depth frames of awkward sizes (tiles of 8 x 4 pixels with rows and columns
left over, single rows and columns) against the same rays integrated through
ohm_integrate_rays, with depths outside the range, NaN and infinite ones; and a
band longer than one piece of the walk.  The TSDF sums are of integers, so both
routes agree bit for bit."""
import math

import numpy as np
import pytest
import torch

from paper_2206_06079_gb300 import ohm, synth, workloads as W
from .parity import assert_maps_identical

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(1, 1), (7, 3), (8, 4), (9, 5), (33, 1), (1, 50), (70, 43), (131, 97)])
@pytest.mark.parametrize("layers,trunc", [(W.TSDF, 0.2), (W.TSDF | W.OCC, 0.13), (W.TSDF, 1.9)])
def test_depth_frame_equals_its_rays(w, h, layers, trunc):
    g = torch.Generator().manual_seed(w * 131 + h)
    s = max(w, h) / 640.0
    K = (525.0 * s, 525.0 * s, (w - 1) / 2.0, (h - 1) / 2.0)
    depth = 0.2 + 5.0 * torch.rand(h, w, generator=g)
    bad = torch.rand(h, w, generator=g)
    depth[bad < 0.02] = 0.0
    depth[(bad >= 0.02) & (bad < 0.04)] = math.nan
    depth[(bad >= 0.04) & (bad < 0.06)] = math.inf
    depth[(bad >= 0.06) & (bad < 0.08)] = 0.3
    depth[(bad >= 0.08) & (bad < 0.10)] = 6.0
    pos, R = synth.camera_pose(5)
    pose = np.concatenate([R.numpy(), pos.numpy()[:, None]], 1)
    # the documented double evaluation
    z = depth.double()
    valid = (z > 0.3) & (z <= 6.0)
    zz = torch.where(valid, z, torch.full_like(z, 6.0)).reshape(-1)
    px = ((torch.arange(w, dtype=torch.float64) - K[2]) / K[0]).expand(h, w).reshape(-1)
    py = ((torch.arange(h, dtype=torch.float64) - K[3]) / K[1])[:, None].expand(h, w).reshape(-1)
    x, y = px * zz, py * zz
    P = torch.from_numpy(pose)
    e = torch.stack([((P[k, 0] * x + P[k, 1] * y) + P[k, 2] * zz) + P[k, 3] for k in range(3)], 1).float()
    f = (~valid).reshape(-1).to(torch.uint8)
    p = W.tsdf_params(layers=layers, tsdf_trunc=trunc, max_rays=w * h, max_regions=512)
    with ohm.Map(**p) as a, ohm.Map(**p) as b:
        for _ in range(2):
            a.integrate_depth(depth.cuda(), K, pose)
            b.integrate(pos.float()[None].cuda(), e.cuda(), f.cuda())
        assert_maps_identical(a, b)
        assert a.stats()["visits"] == b.stats()["visits"] and a.stats()["touched"] == b.stats()["touched"]
