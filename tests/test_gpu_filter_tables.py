"""The consistency filter's two ways to a neighbour's bearing (tables in shared
memory, or computed per pixel) agree bit for bit: many neighbours of different
sizes, whose tables do not fit, against each of them four times in a call of its
own, which tabulates."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_tabulated_bearings_change_nothing():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2211_16266_gb300 as pm
    W, H = 2048, 1023
    rng = np.random.default_rng(5)
    sizes = [(701 + 37 * k, 349 + 11 * k) for k in range(11)] + [(2, 1)]

    def depth(w, h):
        d = rng.uniform(1.9, 2.1, (h, w)).astype(np.float32)
        d[rng.random((h, w)) < 0.1] = 0
        return torch.from_numpy(d).cuda()

    def pose(k):
        a = 0.3 * k
        return np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]]), rng.uniform(-0.01, 0.01, 3)

    ref, rp = depth(W, H), pose(0)
    nbrs, poses = [depth(*s) for s in sizes], [pose(k) for k in range(len(sizes))]
    with pm.Context(0) as ctx:
        kept, together = pm.pmsp_consistency_filter(ctx, ref, rp, nbrs, poses, max_px=12.0, min_views=4)
        apart = torch.zeros_like(together)
        for d, p in zip(nbrs, poses):
            four = pm.pmsp_consistency_filter(ctx, ref, rp, [d] * 4, [p] * 4, max_px=12.0)[1]
            assert bool((four % 4 == 0).all())
            apart += four // 4
        assert bool((together == apart).all()) and 0.2 < float((together > 0).float().mean()) < 1.0
        assert bool((kept == torch.where((ref > 0) & (together >= 4), ref, torch.zeros_like(ref))).all())
