"""Fusion whose first hash table is too small and that comes again with a larger one,
at its end or early (up to 2^23 pixels): every voxel keeps its first pixel. Against a
plain first-of-each-voxel in numpy on the same FP32 points; also at the edges of the
insertion's 32 x 32 tiles and at sizes whose points are written by 1 to 32 blocks a
group of 8192 pixels.
"""
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
    q = np.floor(points * (np.float32(1.0) / np.float32(voxel))).astype(np.int64) + (1 << 20)
    _, first = np.unique((q[:, 0] << 42) | (q[:, 1] << 21) | q[:, 2], return_index=True)
    return np.sort(first)


def _views(sizes, seed):
    rng = np.random.default_rng(seed)
    depths, poses = [], []
    for W, H in sizes:
        d = rng.uniform(0.5, 4.0, (H, W)).astype(np.float32)
        d[rng.random((H, W)) < 0.2] = 0
        a = rng.uniform(-3, 3)
        depths.append(d)
        poses.append((np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]]), rng.uniform(-1, 1, 3)))
    return depths, poses


def _check(pm, ctx, depths, poses, voxel, caps, host=False):
    import torch
    dev = [torch.from_numpy(d).cuda() for d in depths]
    points, origin = [], []
    for k, d in enumerate(dev):  # every valid pixel's point, at a voxel no two of them share
        p, s, n = pm.pmsp_fuse(ctx, [d], [poses[k]], 1e-5)
        assert n == int((depths[k] > 0).sum())
        points.append(p.cpu().numpy())
        origin.append((k << 32) | s.cpu().numpy())
    points, origin = np.concatenate(points), np.concatenate(origin)
    keep = _first_of_voxels(points, voxel)
    for cap in caps:
        p, s, n = pm.pmsp_fuse(ctx, depths if host else dev, poses, voxel, cap and max(1, len(keep) // cap))
        m = len(keep) if cap is None else min(max(1, len(keep) // cap), len(keep))
        p, s = (p, s) if host else (p.cpu().numpy(), s.cpu().numpy())
        assert n == len(keep) and len(p) == m
        assert np.array_equal(s, origin[keep][:m])
        assert np.array_equal(p.view(np.uint32), points[keep][:m].view(np.uint32))
    return len(keep)


@pytest.mark.parametrize("sizes", [[(33, 33), (32, 32), (31, 31)], [(33, 31)], [(64, 65), (31, 33)], [(1, 33)], [(128, 64)],
                                   [(128, 64), (1, 1)], [(700, 350)]])
@pytest.mark.parametrize("voxel", [0.3, 0.01])
def test_tile_edges_and_small_inputs(pm, sizes, voxel):
    depths, poses = _views(sizes, sizes[0][0])
    with pm.Context(0) as ctx:
        _check(pm, ctx, depths, poses, voxel, (None, 1, 3))


# few enough pixels that a table seen to be too small is left early, and too many for that
@pytest.mark.parametrize("sizes", [[(2048, 1024), (2040, 1024)], [(2048, 1024), (2050, 1025), (2047, 1023)]])
@pytest.mark.parametrize("host", [False, True])
def test_a_table_too_small(pm, sizes, host):
    depths, poses = _views(sizes, 5)
    # the first keyframe again, none of whose points is the first of its voxel, and part of the second
    depths += [depths[0], np.where(depths[1] > 2.0, depths[1], np.float32(0))]
    poses += [poses[0], poses[1]]
    assert (sum(d.size for d in depths) <= 1 << 23) == (len(sizes) == 2)
    with pm.Context(0) as ctx:
        n = _check(pm, ctx, depths, poses, 1e-3, (None, 1, 2), host)
        assert n > 3 << 20  # more than three quarters of 2^22 slots
        _check(pm, ctx, depths[:1], poses[:1], 0.05, (None,))  # and a call that the table is large enough for
