"""A backward pass only reads the tape: it leaves the workspace's bytes as they
are, and two passes over one tape may run at once on two streams.  Scenes of a
batch that share an IoR or sigma gradient add up in it."""
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S
from tests.gpu_util import GpuScene

pytestmark = pytest.mark.gpu


def _scene(k, side=64):
    V, F = S.icosphere(3)
    cams = [S.camera((0.3 + 0.2 * k, 0.5, 3.0), (0.0, 0.0, 0.0), (0, 1, 0), 40.0, side, side)]
    return GpuScene(V, F, 1.3 + 0.1 * k, (0.3, 0.1, 0.2), S.sh_env_map(32, 16, k), cams, side, side, 5)


def _item(gs):
    return dt.BatchItem(gs.V, gs.F, gs.bvh, gs.N, gs.ior, gs.sigma, gs.env, gs.cams, gs.width, gs.height, gs.params)


def _near(got, want):
    for x, y in zip(got, want):  # sums of the same terms in another order
        assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max()) + 1e-7


def test_the_workspace_keeps_its_bytes():
    img, tape = _scene(0).render()
    before = tape.ws.buf.clone()
    dt.render_backward(tape, img)
    assert torch.equal(tape.ws.buf, before)
    imgs, tape = dt.render_batch([_item(_scene(k)) for k in range(3)])
    before = tape.ws.buf.clone()
    dt.render_batch_backward(tape, imgs)
    assert torch.equal(tape.ws.buf, before)


def test_two_passes_over_one_tape():
    img, tape = _scene(1, 256).render()
    seeds = [img, 1.0 - 2.0 * img]
    want = [[g.clone() for g in dt.render_backward(tape, s)] for s in seeds]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in seeds]
    for _ in range(10):
        got = []
        for s, seed in zip(streams, seeds):
            with torch.cuda.stream(s):
                got.append(dt.render_backward(tape, seed))
        torch.cuda.synchronize()
        for g, w in zip(got, want):
            _near(g, w)


def test_scenes_that_share_a_gradient_add_up():
    scenes = [_scene(k) for k in range(3)]
    imgs, tape = dt.render_batch([_item(s) for s in scenes])
    alone = dt.render_batch_backward(tape, imgs)
    dior, dsig = torch.full((1,), 7.0, device="cuda"), torch.full((3,), 7.0, device="cuda")
    outs = [(torch.empty_like(s.V), dior, dsig) for s in scenes]
    dt.render_batch_backward(tape, imgs, outs=outs)
    _near([dior, dsig], [sum(a[1] for a in alone), sum(a[2] for a in alone)])
    _near([o[0] for o in outs], [a[0] for a in alone])
