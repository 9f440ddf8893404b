"""Batches on a stream that the caller records.

A captured batch (PMSP_BATCH_GRAPH) is not launched into a recording: the engine's
change flags and plan would go along, and later batches write them. The call
reports the error and the recording goes on. A batch recorded launch by launch
carries no flags: its replay beside a later batch of the same context changes
neither's maps.
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


def _problem(W, H, S, seed):
    import torch
    p = scenes.trajectory_problem(W, H, S, seed_scene=seed, fmt="u8")
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    params = dict(d_min=0.3, d_max=10.0, patch_w=11, patch_stride=2, iterations=6, best_k=min(3, S), sigma_color=0.2,
                  sigma_space=3.0, n_refine=6, neighbor_table=0, seed=9, keyframe_id=seed)
    return (d(p.ref.image), (p.ref.R, p.ref.t), [d(f.image) for f in p.srcs], [(f.R, f.t) for f in p.srcs]), params


def _bits(m):
    return [a.cpu().numpy().view(np.uint32).copy() for a in (m.depth, m.normal, m.cost)]


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("strategy", [0, 1])
def test_a_captured_batch_is_not_recorded(pm, strategy):
    import torch
    prob, params = _problem(256, 128, 3, 77)
    stream = torch.cuda.Stream()
    x = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), pm.Context(0, stream=stream) as ctx:
        batch = pm.Batch([(*prob, params, None)])
        t = pm.pmsp_tuning(0, 0, 0, strategy, 0, 1, 0)
        for _ in range(2):
            pm.pmsp_densify_batch(ctx, batch, pm.PMSP_BATCH_GRAPH, t)
        pm.pmsp_sync(ctx)
        want = _bits(batch.outs[0])
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        x += 1
        with pytest.raises(pm.PmspError):
            pm.pmsp_densify_batch(ctx, batch, pm.PMSP_BATCH_GRAPH, t)
        graph.capture_end()  # the recording holds what else was recorded
        graph.replay()
        batch.outs[0].depth.zero_()
        pm.pmsp_densify_batch(ctx, batch, pm.PMSP_BATCH_GRAPH, t)
        pm.pmsp_sync(ctx)
        assert float(x[0]) == 1.0
        assert _same(_bits(batch.outs[0]), want)


def test_a_recorded_batch_keeps_apart(pm):
    import torch
    first, other = _problem(512, 256, 4, 78), _problem(640, 320, 3, 79)
    stream, beside = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), pm.Context(0, stream=stream) as ctx:
        t = pm.pmsp_tuning(0, 0, 0, 1, 0, 1, 0)
        a, b = pm.Batch([(*first[0], first[1], None)]), pm.Batch([(*other[0], other[1], None)])
        want = []
        for batch in (a, b):
            pm.pmsp_densify_batch(ctx, batch, 0, t)
            pm.pmsp_sync(ctx)
            want.append(_bits(batch.outs[0]))
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        pm.pmsp_densify_batch(ctx, a, 0, t)
        graph.capture_end()
        for batch in (a, b):
            batch.outs[0].depth.zero_()
        stream.synchronize()
        with torch.cuda.stream(beside):
            graph.replay()
        pm.pmsp_densify_batch(ctx, b, 0, t)
        pm.pmsp_sync(ctx)
        beside.synchronize()
        assert _same(_bits(a.outs[0]), want[0]) and _same(_bits(b.outs[0]), want[1])
