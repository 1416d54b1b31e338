"""The TSDF adjoint on a map that no longer holds every region of the frame
(regions moved to the host between the frame and its backward call)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import adjoint
from paper_2206_06079_gb300 import ohm, workloads as W

pytestmark = pytest.mark.gpu

U = 1 << 16
VOXEL, TAU = 0.05, 0.2
CORNERS = [(x, y, z) for x in (0, 1) for y in (0, 1) for z in (0, 1)]  # the regions around (1.6, 1.6, 1.6)
KEPT = {"all": CORNERS, "no middle": [(0, 0, 0), (1, 1, 1)], "no last": CORNERS[:-1], "no first": CORNERS[1:]}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda()


def _frame():
    """A small frame whose bands run from region (0, 0, 0) to (1, 1, 1) through
    the corner that eight regions share."""
    rng = np.random.default_rng(4)
    w, h = 16, 12
    K = (83.0, 83.0, (w - 1) / 2.0, (h - 1) / 2.0)
    z = np.ones(3) / np.sqrt(3.0)
    x = np.array([1.0, -1.0, 0.0]) / np.sqrt(2.0)
    R = np.stack([x, np.cross(z, x), z], 1)
    pose = np.concatenate([R, np.full((3, 1), 0.4)], 1)
    depth = (1.2 * np.sqrt(3.0) + rng.uniform(-0.1, 0.1, size=(h, w))).astype(np.float32)
    depth[0, 0] = 0.0
    return depth, K, pose


def _bands(depth, K, pose):
    """Per pixel: its band's voxels in walk order, s before the clamp, e - c
    in metres, direction and length; (rays of the frame) behind."""
    o, e, f, pt = adjoint.depth_rays(depth, K, pose, 0.3, 6.0)
    scale, cell = U / VOXEL, VOXEL / U
    qo = np.rint(o[0].astype(np.float64) * scale).astype(np.int64)
    out = []
    for ei, fi in zip(e, f):
        if fi:
            out.append(None)
            continue
        qe = np.rint(ei.astype(np.float64) * scale).astype(np.int64)
        d = (qe - qo).astype(np.float64)
        n = np.sqrt((d * d).sum())
        a = qo + np.rint(d * (max(n - TAU * scale, 0.0) / n)).astype(np.int64)
        b = qo + np.rint(d * ((n + TAU * scale) / n)).astype(np.int64)
        v = oracle.walk(a, b)
        r = (qe - (v * U + U // 2)) * cell
        out.append((v, r @ (d / n), r, d / n, n * cell))
    return out, o[0].astype(np.float64), e.astype(np.float64), pt


def _map_with(kept):
    """A map that integrated the frame and holds only the regions `kept`."""
    depth, K, pose = _frame()
    m = ohm.Map(**W.tsdf_params(max_rays=depth.size, max_regions=64, voxel_size=VOXEL, tsdf_trunc=TAU))
    m.integrate_depth(_cuda(depth), K, pose)
    assert m.region_count() == len(CORNERS)
    if len(kept) < len(CORNERS):
        centre = (np.array(kept) + 0.5) * 32 * VOXEL
        m.integrate(_cuda(centre - [0.5, 0, 0]), _cuda(centre))  # bands inside these regions: used last
        m.evict(len(kept))
        assert m.residency() == (len(kept), len(CORNERS) - len(kept))
    return m, depth, K, pose


def _queries(bands):
    """Band voxels of every region and their weights.  Left out: voxels that a
    ray sees within 2e-6 m of the clamp, where float and double s may disagree."""
    rng = np.random.default_rng(5)
    bands = [b for b in bands if b is not None]
    vox = np.unique(np.concatenate([b[0] for b in bands]), axis=0)
    kink = {tuple(v) for b in bands for v in b[0][np.abs(np.abs(b[1]) - TAU) < 2e-6]}
    vox = np.array([v for v in vox.tolist() if tuple(v) not in kink])
    vox = vox[rng.random(len(vox)) < 0.5]
    return vox, rng.normal(size=len(vox)).astype(np.float32)


def test_missing_regions_leave_the_map_usable():
    m, depth, K, pose = _map_with(KEPT["no middle"])
    vox, g = _queries(_bands(depth, K, pose)[0])
    m.tsdf_backward(_cuda(depth), K, pose, _cuda((vox + 0.5) * VOXEL), _cuda(g))
    m.sync()
    end = np.array([[0.8, 0.8, 0.8]])
    before = m.query(_cuda(end), tsdf=True)["tsdf"][0, 1].item()
    m.integrate(_cuda(end - [0.5, 0, 0]), _cuda(end))
    assert m.query(_cuda(end), tsdf=True)["tsdf"][0, 1].item() == before + 1


@pytest.mark.parametrize("kept", list(KEPT))
def test_gradient_up_to_the_first_missing_region(kept):
    """Each ray's band counts up to its first voxel in a missing region, as
    the sum over its unclamped voxels in float64 (1e-3 relative: the kernel's s
    and chain rule are float32)."""
    m, depth, K, pose = _map_with(KEPT[kept])
    bands, o, e, pt = _bands(depth, K, pose)
    vox, g = _queries(bands)
    gd, gt = m.tsdf_backward(_cuda(depth), K, pose, _cuda((vox + 0.5) * VOXEL), _cuda(g))
    m.sync()
    weight = {tuple(v): float(x) for v, x in zip(vox.tolist(), g)}
    held = set(KEPT[kept])
    at = {}
    for b in bands:
        for v in ([] if b is None else b[0].tolist()):
            at[tuple(v)] = None
    w = m.query(_cuda((np.array(list(at)) + 0.5) * VOXEL), tsdf=True)["tsdf"][:, 1].cpu().numpy().astype(np.float64)
    at = dict(zip(at, w))
    ge, go = np.zeros((len(e), 3)), np.zeros(3)
    cut = 0
    for j, b in enumerate(bands):
        if b is None:
            continue
        A, B = 0.0, np.zeros(3)
        for v, s, r in zip(b[0].tolist(), b[1], b[2]):
            if tuple(c >> 5 for c in v) not in held:
                cut += 1
                break
            if abs(s) < TAU and tuple(v) in weight:
                wv = weight[tuple(v)] / at[tuple(v)]
                A += wv
                B += wv * (r - s * b[3])
        ge[j] = A * b[3] + B / b[4]
        go -= B / b[4]
    assert (cut > 0) == (kept != "all")
    gz, twist = adjoint.chain_to_depth_and_twist(ge, go, e, o, pose[:, :3], pt)
    gd = gd.cpu().numpy().reshape(-1).astype(np.float64)
    assert np.abs(gz).max() > 0
    assert (np.abs(gd - gz) <= 1e-3 * np.abs(gz) + 1e-6 * np.abs(gz).max()).all(), np.abs(gd - gz).max()
    assert np.linalg.norm(gt.cpu().numpy() - twist) <= 1e-3 * np.linalg.norm(twist)
