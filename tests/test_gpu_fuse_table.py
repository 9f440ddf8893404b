"""Fusion where its hash table starts too small, and at tile edges, against a
plain first-of-each-voxel in numpy on the same FP32 points."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2211_16266_gb300 as pm
    return pm


def _first_of_voxels(points, voxel):
    q = np.floor(points * (np.float32(1.0) / np.float32(voxel))).astype(np.int64)
    _, first = np.unique(q, axis=0, return_index=True)
    return np.sort(first)


@pytest.mark.parametrize("sizes,voxel", [
    ([(64, 32)], 1e-3),                    # every pixel a voxel of its own
    ([(640, 320), (333, 167)], 2e-3),
    ([(2048, 1024), (2048, 1024)], 1e-3),  # more voxels than a table within L2 takes: it grows
    ([(33, 9), (32, 8), (31, 7)], 0.05),   # edges of the 32 x 8 tiles
    ([(1, 1)], 0.02), ([(257, 1), (1, 65)], 0.2),
    ([(320, 160)] * 16, 0.5),              # many pixels to a voxel, the most keyframes
])
@pytest.mark.parametrize("host", [False, True])
def test_fuse_equals_first_of_each_voxel(pm, sizes, voxel, host):
    import torch
    rng = np.random.default_rng(len(sizes) * 1000 + sizes[0][0])
    depths, poses = [], []
    for W, H in sizes:
        d = rng.uniform(0.5, 4.0, (H, W)).astype(np.float32)
        d[rng.random((H, W)) < 0.2] = 0
        depths.append(d)
        a = rng.uniform(-3, 3)
        poses.append((np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]]), rng.uniform(-1, 1, 3)))
    dev = [torch.from_numpy(d).cuda() for d in depths]
    with pm.Context(0) as ctx:
        # every valid pixel's point: one keyframe at a time at a voxel no two of its points share, else the finest there is
        points, origin = [], []
        for k, d in enumerate(dev):
            p, s, n = pm.pmsp_fuse(ctx, [d], [poses[k]], 1e-5)
            assert n == int((depths[k] > 0).sum())
            points.append(p.cpu().numpy())
            origin.append((k << 32) | s.cpu().numpy())
        points, origin = np.concatenate(points), np.concatenate(origin)
        keep = _first_of_voxels(points, voxel)
        for cap in (None, len(keep), max(1, len(keep) // 3)):
            p, s, n = pm.pmsp_fuse(ctx, depths if host else dev, poses, voxel, cap)
            m = len(keep) if cap is None else min(cap, len(keep))
            p, s = (p, s) if host else (p.cpu().numpy(), s.cpu().numpy())
            assert n == len(keep) and len(p) == m
            assert np.array_equal(s, origin[keep][:m])
            assert np.array_equal(p.view(np.uint32), points[keep][:m].view(np.uint32))
