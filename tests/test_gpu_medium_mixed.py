"""A batch whose warps march several media at once: hash textures of different
depth, dense grids, scenes without a medium, and boxes that hold the object or
cut it, so that a warp's lanes leave its loops at different levels and need
different forms of the walk.  Images and all gradients are those of each scene
rendered alone, on a full tape and on one with the medium's moments."""
import re
from pathlib import Path

import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S


def test_votes_name_their_lanes():
    # the lanes of __activemask() need not be converged at the vote that takes it
    for f in (Path(dt.__file__).parent / "csrc").iterdir():
        assert not re.search(r"_sync\(\s*__activemask", f.read_text()), f.name


def _item(k, side, moments):
    dev = torch.device("cuda:0")
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x, np.float32)).to(dev)  # noqa: E731
    V, F = S.icosphere(3)
    V, F = t(V), torch.from_numpy(F).to(dev)
    cam = S.camera((0.3, 0.5 + 0.1 * k, 3.0), (0.0, 0.0, 0.0), (0, 1, 0), 40.0, side, side)
    half = (1.25, 0.7)[k % 2]  # the box holds the sphere, or cuts it
    ramp = torch.linspace(0.0, 1.0, 1 << 12, device=dev)
    med = None
    if k in (0, 1, 5):  # smooth values: unrelated entries make a few rays dominate the IoR gradient
        levels = (5, 2, 1)[min(k, 2)]
        table = torch.stack([ramp, 1.0 - ramp, 0.5 * ramp], 1)[None].repeat(levels, 1, 1) / levels
        med = dt.HashTexture(table.contiguous(), [6 + 3 * l for l in range(levels)], (-half,) * 3, (half,) * 3, 0.07)
    elif k in (2, 3):
        n = 9 + k
        g = torch.linspace(0.0, 1.0, n, device=dev)
        mu = torch.stack(torch.meshgrid(g, g * g, 1.0 - g, indexing="ij"), 3)
        med = dt.Medium(mu.contiguous(), (-half,) * 3, (half,) * 3, 0.05)
    return dt.BatchItem(V, F, dt.build_bvh(V, F), dt.vertex_normals(V, F), torch.tensor([1.3], device=dev),
                        t([0.2, 0.1, 0.3]), t(S.sh_env_map(32, 16, k)), t(cam.as_array()[None]), side, side,
                        dt.Params(5, moments=moments), medium=med)


@pytest.mark.gpu
@pytest.mark.parametrize("moments", [False, True])
def test_a_batch_of_several_media(moments):
    items = [_item(k, 40 + k, moments) for k in range(6)]
    imgs, tape = dt.render_batch(items)
    grads = dt.render_batch_backward(tape, [i + 0.5 for i in imgs], env_grad=True)
    for it, img, got in zip(items, imgs, grads):
        one, t1 = dt.render(it.V, it.F, it.bvh, it.N, it.ior, it.sigma, it.env, it.cams, it.width, it.height, it.params,
                            medium=it.medium)
        want = dt.render_backward(t1, one + 0.5, env_grad=True)
        assert len(got) == len(want)
        for x, y in zip((img, *got), (one, *want)):  # sums of the same terms in another order
            assert float((x - y).abs().max()) <= 1e-4 * float(y.abs().max()) + 1e-6
