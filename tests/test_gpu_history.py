"""Whole runs against the same run driven step by step, bit for bit.

Within a run the half-sweeps leave out neighbour candidates that were already
tried (PixelParams::changed), and on larger keyframes drop refinement tests that
provably cannot win (sweep_bounded); a half-sweep called on its own has no history and
tries them all. Both must give the same maps: in one call, warped, batched by
either strategy, replayed from a graph, and recorded by the caller.
"""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2211_16266_gb300 as pm
    return pm


FORMS = [  # W, H, views, format, window, stride, table, best_k, n_refine
    (96, 48, 1, "u8", 11, 2, 0, 1, 6), (66, 34, 2, "f16", 7, 1, 1, 1, 6), (250, 130, 3, "f32", 9, 3, 1, 2, 6),
    (8, 4, 2, "u8", 5, 1, 0, 2, 6), (128, 64, 6, "u8", 11, 2, 0, 3, 6), (100, 52, 7, "f32", 11, 2, 1, 7, 0),
    (64, 34, 10, "f16", 5, 2, 0, 4, 9), (64, 32, 12, "u8", 3, 1, 0, 3, 2), (70, 36, 16, "u8", 21, 5, 0, 16, 1),
    # from 456 tiles on: the refinement tests dropped by a bound, in every window class, ragged, with more tests
    # than are drawn ahead, with none, with no bilateral weights and with the mean over all views
    (518, 250, 4, "u8", 11, 2, 0, 1, 6), (512, 256, 5, "f16", 7, 1, 1, 5, 9), (640, 200, 6, "f32", 9, 3, 0, 3, 6),
    (512, 258, 6, "f32", 9, 2, 0, 3, 6), (514, 258, 7, "u8", 11, 2, 1, 2, 0), (512, 260, 10, "u8", 11, 2, 0, 3, 30),
]


def _problem(form, n_iter):
    W, H, S, fmt, pw, st, table, k, nr = form
    p = scenes.trajectory_problem(W, H, S, seed_scene=1020 + S, fmt=fmt)
    params = dict(d_min=0.3, d_max=10.0, patch_w=pw, patch_stride=st, iterations=n_iter, best_k=k,
                  sigma_color=0.0 if S == 5 else 0.2, sigma_space=0.0 if S == 5 else 3.0, n_refine=nr, neighbor_table=table, seed=9, keyframe_id=S)
    import torch
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return (d(p.ref.image), (p.ref.R, p.ref.t), [d(f.image) for f in p.srcs], [(f.R, f.t) for f in p.srcs]), params


def _steps(pm, ctx, prob, params, start=None):
    m = start if start is not None else pm.pmsp_init(ctx, *prob, params)
    for it in range(params["iterations"]):
        for colour in range(2):
            pm.pmsp_halfsweep(ctx, *prob, params, colour, it, m)
    return _bits(pm, ctx, m)


def _bits(pm, ctx, m):
    pm.pmsp_sync(ctx)
    return [a.cpu().numpy().view(np.uint32).copy() for a in (m.depth, m.normal, m.cost)]


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


# one, two, four and eight lanes a pixel (by size and view count): the same maps with one, in the shapes and the
# company that get one, and in the persistent kernel
LANE_FORMS = [(64, 32, 2, "u8", 7, 1, 0, 1, 6), (8, 4, 1, "f32", 5, 1, 0, 1, 5), (130, 66, 6, "f16", 11, 2, 1, 3, 7),
              (256, 128, 2, "u8", 7, 1, 0, 1, 6), (250, 130, 3, "f32", 9, 3, 1, 2, 13), (256, 130, 6, "u8", 11, 2, 0, 3, 6),
              (322, 158, 4, "f16", 11, 2, 0, 4, 1), (384, 194, 2, "u8", 13, 2, 0, 2, 0), (66, 34, 16, "u8", 5, 1, 0, 7, 6)]


@pytest.mark.parametrize("form", LANE_FORMS)
def test_lanes_per_pixel_change_nothing(pm, form):
    prob, params = _problem(form, 4)
    with pm.Context(0) as ctx:
        want = _steps(pm, ctx, prob, params)
        assert _same(_bits(pm, ctx, pm.pmsp_densify(ctx, *prob, params)), want)
        # a tile shape asked for is served by one lane a pixel (11x11 / 2 and 7x7 windows), and so is a keyframe in a crowd
        for tile, n in ((1, 1), (0, 1 if form[0] > 300 else 60)):
            batch = pm.Batch([(*prob, params, None)] * n)
            pm.pmsp_densify_batch(ctx, batch, 0, pm.pmsp_tuning(0, 0, 0, 1, tile, 1, 0))
            for out in batch.outs[::max(1, n // 3)]:
                assert _same(_bits(pm, ctx, out), want)
        batch = pm.Batch([(*prob, params, None)])
        pm.pmsp_densify_batch(ctx, batch, 0, pm.pmsp_tuning(0, 0, 0, 0, 0, 1, 0))
        if form[2] <= 10:  # (above, the persistent kernel scores view by view)
            assert _same(_bits(pm, ctx, batch.outs[0]), want)


@pytest.mark.parametrize("form", FORMS)
def test_run_equals_its_steps(pm, form):
    import torch
    prob, params = _problem(form, 5)
    with pm.Context(0) as ctx:
        want = _steps(pm, ctx, prob, params)
        for _ in range(2):  # the second run finds the first one's flags
            assert _same(_bits(pm, ctx, pm.pmsp_densify(ctx, *prob, params)), want)
        prev = pm.Maps(*[torch.from_numpy(a.view(np.float32)).cuda() for a in want])
        pose = (np.eye(3), np.array([0.05, 0.0, 0.02]))
        first = pm.pmsp_warp_init(ctx, *prob, params, prev, pose)
        warped = _steps(pm, ctx, prob, params, first)
        assert _same(_bits(pm, ctx, pm.pmsp_densify_warped(ctx, *prob, params, prev, pose)), warped)


def test_batches_equal_their_steps(pm):
    import torch
    probs = [_problem(FORMS[k], 3 + k % 3) for k in (0, 2, 4, 5, 6, 9, 12)]
    with pm.Context(0) as ctx:
        want = [_steps(pm, ctx, *p) for p in probs]
        for strategy in (0, 1):
            for flags in (0, pm.PMSP_BATCH_GRAPH):
                batch = pm.Batch([(*p, params, None) for p, params in probs])
                t = pm.pmsp_tuning(0, 0, 0, strategy, 0, 1, 0)
                for _ in range(3):  # eager, captured, replayed
                    pm.pmsp_densify_batch(ctx, batch, flags, t)
                for out, w in zip(batch.outs, want):
                    assert _same(_bits(pm, ctx, out), w)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), pm.Context(0, stream=stream) as ctx:  # a run recorded by the caller
        prob, params = probs[2]
        out = pm.pmsp_densify(ctx, *prob, params)
        pm.pmsp_sync(ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            pm.pmsp_densify(ctx, *prob, params, out)
        # a larger reference against the same sources moves the context's flags (the
        # recording keeps the source textures, so their sizes stay)
        big = torch.rand(128, 256, device="cuda")
        other = pm.pmsp_densify(ctx, big, *prob[1:], params)
        out.depth.zero_()
        graph.replay()
        stream.synchronize()
        assert _same(_bits(pm, ctx, out), want[2])
        assert float(other.depth.min()) > 0
