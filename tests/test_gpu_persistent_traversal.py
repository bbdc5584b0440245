"""The persistent traversal (more than 40,960 camera rays): on the coded binary
nodes, on the exact ones of a scene whose detailed part the codes cannot resolve,
and in a batch of both; in append order and in bucket order; on a full tape and
on a checkpointed one, whose hits are a ring of two levels.  The order changes
nothing that is traced, a batch's scenes keep their own kind of nodes, and an
unresolved part costs no more triangle tests than float boxes do."""
import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S
from tests.gpu_util import GpuScene, segments_by_key

pytestmark = pytest.mark.gpu

W, H, VIEWS = 48, 40, 22  # 42,240 camera rays a scene


def _scene(kind, checkpoint=False):
    if kind == "resolved":
        V, F = S.two_tori_mesh(36)
        cams, t_min = S.fibonacci_views(VIEWS, 3.0, W, H), 1e-5
    elif kind == "ground":  # few triangles, and one 1e5 times their size
        V, F = S.icosphere(1)
        V = np.concatenate([V, np.float32([[-1e5, -2, -1e5], [1e5, -2, -1e5], [0, -2, 1e5]])])
        F = np.concatenate([F, np.int32([[len(V) - 3, len(V) - 1, len(V) - 2]])])
        cams, t_min = [S.camera((0.3 + 0.01 * k, 0.5, 3.0), (0, 0, 0), (0, 1, 0), 45.0, W, H) for k in range(VIEWS)], 1e-5
    else:  # a large sphere, and beside it a small one with edges of two steps of the codes' grid
        scale = 1e-3
        V, F = S.icosphere(2)
        v, f = S.icosphere(4)
        V, F = np.concatenate([V, v * scale + np.float32([1.5, 0, 0])]), np.concatenate([F, f + len(V)])
        eyes = [(1.5 + 3 * scale * np.sin(a), scale * np.cos(2 * a), 3 * scale * np.cos(a)) for a in np.arange(VIEWS)]
        cams, t_min = [S.camera(e, (1.5, 0.0, 0.0), (0, 1, 0), 40.0, W, H) for e in eyes], 1e-8
    gs = GpuScene(V, F, 1.4, (0.3, 0.1, 0.2), S.sh_env_map(32, 16, 0), cams, W, H, 6, t_min=t_min)
    p = gs.params
    gs.params = dt.Params(p.max_depth, t_min=t_min, checkpoint=checkpoint)
    return gs


def _item(gs):
    return dt.BatchItem(gs.V, gs.F, gs.bvh, gs.N, gs.ior, gs.sigma, gs.env, gs.cams, gs.width, gs.height, gs.params)


def _run(scenes, order):
    old = dt.set_tuning(order_min_rays=0, trace_order=order)
    try:
        g = torch.Generator("cuda").manual_seed(1)
        if len(scenes) == 1:
            img, tape = scenes[0].render()
            seeds = [torch.randn(img.shape, generator=g, device="cuda")]
            return [img], tape.stats, [dt.render_backward(tape, seeds[0])]
        imgs, tape = dt.render_batch([_item(s) for s in scenes])
        seeds = [torch.randn(i.shape, generator=g, device="cuda") for i in imgs]
        return imgs, tape.stats, dt.render_batch_backward(tape, seeds)
    finally:
        dt.set_tuning(**old)


STATS = ("segments", "level_count", "hits", "misses", "tir", "nodes_visited", "tris_tested")


@pytest.mark.parametrize("checkpoint", [False, True])
@pytest.mark.parametrize("kinds", [["resolved"], ["unresolved"], ["resolved", "unresolved"], ["resolved", "resolved"]])
def test_the_order_changes_nothing(kinds, checkpoint):
    scenes = [_scene(k, checkpoint) for k in kinds]
    i0, s0, g0 = _run(scenes, 0)
    i1, s1, g1 = _run(scenes, 20)
    assert s0["status"] == s1["status"] == dt.DT_OK
    for key in STATS:
        assert s0[key] == s1[key], key
    for a, b in zip(i0, i1):
        np.testing.assert_allclose(b.cpu().numpy(), a.cpu().numpy(), rtol=1e-6, atol=1e-6)
    for a, b in zip(g0, g1):  # sums of the same terms in another order
        for x, y in zip(a, b):
            x, y = x.cpu().numpy().astype(np.float64), y.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(x - y) <= 1e-4 * np.linalg.norm(x) + 1e-8


def test_a_batch_traces_each_scene_with_its_own_nodes():
    scenes = [_scene("resolved"), _scene("unresolved")]
    alone = [_run([s], 20) for s in scenes]
    imgs, stats, _ = _run(scenes, 20)
    for key in ("segments", "hits", "nodes_visited", "tris_tested"):
        assert stats[key] == sum(a[1][key] for a in alone), key
    for a, img in zip(alone, imgs):
        np.testing.assert_allclose(img.cpu().numpy(), a[0][0].cpu().numpy(), rtol=1e-6, atol=1e-6)


@pytest.mark.parametrize("kind", ["unresolved", "ground"])
def test_an_unresolved_part_costs_what_float_boxes_do(kind):
    gs = _scene(kind)
    got = {}
    for width in (2, 4):
        old = dt.set_tuning(bvh_width=width)
        try:
            _, tape = gs.render()
        finally:
            dt.set_tuning(**old)
        si, sf = dt.dump_segments(tape)
        got[width] = (tape.stats, segments_by_key(si[si[:, 0] < W * H].cpu().numpy()))
    assert got[2][1] == got[4][1]
    assert got[2][0]["tris_tested"] <= 1.25 * got[4][0]["tris_tested"]
    # arbitrary rays: the camera rays, asked again
    si, sf = dt.dump_segments(tape)
    cam = si[:, 1] == 1
    tri, tbb = dt.closest_hit(gs.bvh, sf[cam][:, 3:6].contiguous(), sf[cam][:, 6:9].contiguous(),
                              t_min=gs.params.t_min)
    assert torch.equal(tri, si[cam][:, 2]) and torch.equal(tbb, sf[cam][:, :3])
