"""The consistency filter at widths around its 32-pixel strips and at map sizes that
start it in blocks of one warp to sixteen, against FP64, and with bearing tables
between 48 KB and the largest that it takes (72 KB), against the form that computes
the bearings.

FP64 decides a neighbour alike unless a column or row lies within EDGE of rounding
to another pixel or the distance within EDGE of the threshold; EDGE is ten times
the FP32 error of two projections (1e-6 rad each at W / 2 pi pixels per radian, of
points whose distance from either camera is at least half their range), at W = 1100.
A column's error grows towards the poles by 1 / cos(latitude).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EDGE = 10 * 2 * 1e-6 * 1100 / (2 * np.pi) * 2


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2211_16266_gb300 as pm
    return pm


def _pose(k, rng):
    a = 0.3 * k
    return np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]]), rng.uniform(-0.01, 0.01, 3)


def _depth(w, h, rng):
    d = rng.uniform(1.9, 2.1, (h, w)).astype(np.float32)
    d[rng.random((h, w)) < 0.1] = 0
    return d


def _bearing(u, v, W, H):
    lon, lat = 2 * np.pi * (u + 0.5) / W - np.pi, np.pi / 2 - np.pi * (v + 0.5) / H
    return np.stack([np.cos(lat) * np.sin(lon), -np.sin(lat), np.cos(lat) * np.cos(lon)])


def _project(X, W, H):
    lon, lat = np.arctan2(X[0], X[2]), np.arctan2(-X[1], np.hypot(X[0], X[2]))
    return W * (lon + np.pi) / (2 * np.pi) - 0.5, H * (np.pi / 2 - lat) / np.pi - 0.5


def _edge(X):
    return EDGE * np.sqrt((X * X).sum(0)) / np.maximum(np.hypot(X[0], X[2]), 1e-6)


def _near_half(x, edge):
    return ~(np.abs(x + 0.5 - np.round(x + 0.5)) >= edge)


def _reference(d, pose, nbrs, poses, max_px):
    """Agreeing neighbours of every pixel, and how many of its decisions are too close to call."""
    H, W = d.shape
    v, u = np.mgrid[:H, :W].astype(np.float64)
    X = d * _bearing(u, v, W, H)
    agree, unsure = np.zeros((H, W), int), np.zeros((H, W), int)
    for dn, (Rn, tn) in zip(nbrs, poses):
        h, w = dn.shape
        R = Rn @ pose[0].T
        t = tn - R @ pose[1]
        Y = np.einsum("ij,jhw->ihw", R, X) + t[:, None, None]
        uc, vc = _project(Y, w, h)
        ui, vi = np.floor(uc + 0.5).astype(int) % w, np.clip(np.floor(vc + 0.5).astype(int), 0, h - 1)
        dj = dn[vi, ui].astype(np.float64)
        Z = np.einsum("ij,jhw->ihw", R.T, dj * _bearing(ui, vi, w, h) - t[:, None, None])
        u2, v2 = _project(Z, W, H)
        du = u2 - u
        du -= W * np.floor(du / W + 0.5)  # (at half a panorama either way gives the same distance)
        dist = np.hypot(du, v2 - v)
        agree += (d > 0) & (dj > 0) & (dist < max_px)
        with np.errstate(invalid="ignore"):
            far = (dj > 0) & ~(np.abs(dist - max_px) >= _edge(Z))
            unsure += _near_half(uc, _edge(Y)) | _near_half(vc, EDGE) | far
    return agree, np.where(d > 0, unsure, 0)


@pytest.mark.parametrize("W,H", [(2, 1), (31, 9), (32, 16), (33, 17), (63, 40), (130, 66), (511, 20), (514, 257), (1026, 130)])
@pytest.mark.parametrize("n", [1, 4, 7])
def test_strips_against_fp64(pm, W, H, n):
    import torch
    rng = np.random.default_rng(W * 10 + n)
    sizes = [(W, H) if k % 2 == 0 else (W + 3 + k, H + k) for k in range(n)]
    d, nbrs = _depth(W, H, rng), [_depth(*s, rng) for s in sizes]
    pose, poses = _pose(0, rng), [_pose(k + 1, rng) for k in range(n)]
    want, unsure = _reference(d, pose, nbrs, poses, 2.0)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    with pm.Context(0) as ctx:
        kept, agree = pm.pmsp_consistency_filter(ctx, dev(d), pose, [dev(x) for x in nbrs], poses, max_px=2.0, min_views=2)
        kept, agree = kept.cpu().numpy(), agree.cpu().numpy()
    assert (np.abs(agree - want) <= unsure).all()
    assert W * H < 500 or (unsure == 0).mean() > 0.5
    assert np.array_equal(kept, np.where((d > 0) & (agree >= 2), d, np.float32(0)))


# reference, neighbours that leave the tables within 72 KB, one more size that takes them beyond
@pytest.mark.parametrize("ref,within,beyond", [
    ((3840, 1920), [(512, 256)] * 4, (2048, 1024)),  # 52 KB, then 77
    ((4096, 2048), [(2048, 1024)], (2, 1)),          # 72 KB exactly, then 3 entries more
    ((3840, 1920), [(2048, 1024)], (512, 256)),      # 71 KB, then 77
])
def test_large_tables_change_nothing(pm, ref, within, beyond):
    import torch
    rng = np.random.default_rng(ref[0] + len(within))
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    d, pose = dev(_depth(*ref, rng)), _pose(0, rng)
    nbrs, poses = [dev(_depth(*s, rng)) for s in within], [_pose(k + 1, rng) for k in range(len(within))]
    more, more_pose = dev(_depth(*beyond, rng)), _pose(6, rng)
    with pm.Context(0) as ctx:
        agree = lambda n, p: pm.pmsp_consistency_filter(ctx, d, pose, n, p, max_px=12.0)[1]  # noqa: E731
        tabulated, alone = agree(nbrs, poses), agree([more], [more_pose])
        direct = agree(nbrs + [more], poses + [more_pose])
        assert bool((direct == tabulated + alone).all())
        assert 0.2 < float((tabulated > 0).float().mean()) < 1.0
