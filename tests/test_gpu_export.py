"""Region export: every layer equals point queries of the same voxels and the
oracle's dense export, for single regions, ranges that start mid-pool, regions
with and without samples, and output pointers on and off 16-byte boundaries."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2206_06079_gb300 import ohm, synth, workloads as W
from .parity import compare_dense, compare_ndt

pytestmark = pytest.mark.gpu

ALL = W.OCC | W.NDT | W.TSDF | W.COUNTS | W.DECAY | W.MEAN
SHAPES = dict(occupancy=(torch.float32, 1), counts=(torch.int32, 2), ndt=(torch.int64, 10), tsdf=(torch.float32, 2),
              path_sum=(torch.int64, 1), mean=(torch.int64, 1))
ORDER = ("occupancy", "counts", "ndt", "tsdf", "path_sum", "mean")


def _export_at(gm, first, count, shift):
    """Export into views `shift` elements into their storage."""
    out, args = {}, []
    for name in ORDER:
        dtype, width = SHAPES[name]
        buf = torch.full((shift + count * ohm.REGION_VOXELS * width + 3,), 77, dtype=dtype, device="cuda")
        out[name] = buf
        args.append(ctypes.c_void_p(buf.data_ptr() + shift * buf.element_size()))
    keys = torch.empty((count, 3), dtype=torch.int32, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    code = ohm.load_library().ohm_map_export(gm.handle, first, count, ctypes.c_void_p(keys.data_ptr()), *args, stream)
    assert code == ohm.OK
    torch.cuda.synchronize()
    res = {"keys": keys}
    for name in ORDER:
        n = count * ohm.REGION_VOXELS * SHAPES[name][1]
        b = out[name]
        assert bool((b[:shift] == 77).all()) and bool((b[shift + n:] == 77).all())  # nothing written outside
        res[name] = b[shift:shift + n]
    return res


def test_export_alignment_ranges_and_oracle():
    rays = synth.room_scan(n=6000)
    o, e, f = rays.numpy()
    f[::7] = 1
    p = W.room_params(layers=ALL, max_regions=128, max_ndt_regions=128, max_rays=6000)
    with ohm.Map(**p) as gm:
        om = oracle.OracleMap(**W.oracle_params(p))
        for _ in range(2):
            gm.integrate(o, e, f)
            om.integrate(o, e, f)
        n = compare_dense(gm, om, tsdf=True, path=True, mean=True)
        compare_ndt(gm, om)
        for first, count in ((0, n), (n // 2, 1), (n - 3, 3)):
            a = _export_at(gm, first, count, 0)
            for shift in (1, 2):
                b = _export_at(gm, first, count, shift)
                for name in a:
                    assert torch.equal(a[name].view(torch.uint8), b[name].view(torch.uint8)), (name, shift, first)
        # a released slot and one never used export as unobserved
        x = gm.export(ndt=True, tsdf=True, first=120, count=4)
        assert bool(torch.isnan(x["occupancy"]).all()) and not bool(x["ndt"].any()) and not bool(x["tsdf"].any())
        assert np.array_equal(a["keys"].cpu().numpy(), gm.export(first=n - 3, count=3)["keys"].cpu().numpy())
