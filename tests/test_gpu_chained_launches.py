"""The kernels of a pass are launched before their predecessors have ended and
wait for them on the device.  Renders and gradients of changing inputs, back to
back on one stream and on several at once without a synchronisation between
them, and replayed from a captured graph, are those of passes that the host has
waited for, one by one."""
import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S
from tests.gpu_util import GpuScene

pytestmark = pytest.mark.gpu


def _scenes(n):
    out = []
    for k in range(n):
        V, F = S.icosphere(2)
        cam = S.camera((0.3 + 0.1 * k, 0.5, 3.0), (0.0, 0.0, 0.0), (0, 1, 0), 40.0, 40, 36)
        out.append(GpuScene(V * np.float32(1.0 + 0.1 * k), F, 1.3 + 0.05 * k, (0.3, 0.1, 0.2), S.sh_env_map(32, 16, k),
                            [cam], 40, 36, 5))
    return out


def _pass(gs, ws, out, stream=None):
    """Forward and gradient with the squared image's weight; no host wait."""
    img, tape = dt.render(gs.V, gs.F, gs.bvh, gs.N, gs.ior, gs.sigma, gs.env, gs.cams, gs.width, gs.height, gs.params,
                          ws=ws, out=out, stream=stream, check=False)
    return img, dt.render_backward(tape, img, stream=stream)


def _near(got, want):
    # sums of the same terms in another order
    for x, y in zip(got, want):
        assert float((x - y).abs().max()) <= 1e-4 * float(y.abs().max()) + 1e-6


def _reference(scenes):
    ref = []
    for gs in scenes:
        img, tape = gs.render()
        torch.cuda.synchronize()
        grads = dt.render_backward(tape, img)
        torch.cuda.synchronize()
        ref.append([img.clone()] + [g.clone() for g in grads])
    return ref


def test_passes_back_to_back_share_a_workspace():
    scenes = _scenes(4)
    ref = _reference(scenes)
    ws = dt.Workspace(40 * 40 * 36, torch.device("cuda:0"))
    outs = [torch.empty(1, 36, 40, 3, device="cuda") for _ in scenes]
    got = []
    for _ in range(5):
        got = [_pass(gs, ws, o) for gs, o in zip(scenes, outs)]
    torch.cuda.synchronize()
    for (img, grads), want in zip(got, ref):
        _near([img, *grads], want)


def test_passes_on_several_streams():
    scenes = _scenes(4)
    ref = _reference(scenes)
    outs = [torch.empty(1, 36, 40, 3, device="cuda") for _ in scenes]
    streams = [torch.cuda.Stream() for _ in scenes]
    torch.cuda.synchronize()
    got = [None] * 4
    for _ in range(5):
        for k, gs in enumerate(scenes):
            with torch.cuda.stream(streams[k]):
                got[k] = _pass(gs, None, outs[k])
    torch.cuda.synchronize()
    for (img, grads), want in zip(got, ref):
        _near([img, *grads], want)


def test_captured_passes():
    gs = _scenes(1)[0]
    want = gs.render()[0].clone()
    ws = dt.Workspace(40 * 40 * 36, torch.device("cuda:0"))
    out = torch.empty(1, 36, 40, 3, device="cuda")

    def run():
        return dt.render(gs.V, gs.F, gs.bvh, gs.N, gs.ior, gs.sigma, gs.env, gs.cams, gs.width, gs.height, gs.params,
                         ws=ws, out=out, check=False)

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        run()
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
        run()
    out.fill_(-1.0)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    _near([out], [want])
    gs.ior.fill_(1.2)  # replays read the scene anew
    graph.replay()
    torch.cuda.synchronize()
    _near([out], [gs.render()[0]])
    assert float((out - want).abs().max()) > 1e-3


def test_captured_build_and_refit():
    V, F = S.icosphere(4)  # more triangles than one small task of the builder
    V, F = torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda()
    o = torch.randn(2000, 3, device="cuda") * 3.0
    d = -o / o.norm(dim=1, keepdim=True)
    built, refitted = dt.build_bvh(V, F), dt.build_bvh(V, F)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        built.build(V, F)
        refitted.refit(V, F)
        N = dt.vertex_normals(V, F)
    for scale in (0.7, 1.2):
        V.mul_(scale)  # replays read the vertices anew
        graph.replay()
        want = dt.closest_hit(dt.build_bvh(V, F), o, d)
        for bvh in (built, refitted):
            got = dt.closest_hit(bvh, o, d)
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        assert torch.equal(N, dt.vertex_normals(V, F))
