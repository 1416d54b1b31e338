"""The prepare kernel's two block sizes: calls that fit one wave of the device
(four blocks of 256 per SM) go out in blocks of 128 rays, larger ones in blocks
of 256.  Both ends of that line, partial last blocks and the smallest calls
must give the oracle's regions, log-odds, counts and NDT moments exactly."""
import numpy as np
import pytest
import torch

import oracle
from paper_2206_06079_gb300 import ohm, workloads as W
from .parity import compare_dense, compare_ndt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 257, "wave-127", "wave", "wave+1", "wave+129"])
def test_both_block_sizes_match_the_oracle(n):
    if isinstance(n, str):
        wave = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 256
        n = wave + int(n[4:] or 0)
    rng = np.random.default_rng(n)
    o = np.array([[0.21, -0.37, 0.11]], np.float32)
    e = (o + rng.standard_normal((n, 3)) * np.array([1.5, 1.2, 0.4])).astype(np.float32)
    f = (rng.random(n) < 0.2).astype(np.uint8)
    p = W.room_params(layers=W.OCC | W.COUNTS | W.NDT, max_regions=512, max_ndt_regions=512, max_rays=max(n, 1024))
    with ohm.Map(**p) as gm:
        om = oracle.OracleMap(**W.oracle_params(p))
        gm.integrate(o, e, f)
        om.integrate(o, e, f)
        assert compare_dense(gm, om) > 0
        compare_ndt(gm, om)
