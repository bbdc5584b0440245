"""Batches of other scenes, other numbers of scenes and other hash textures,
back to back in one workspace: a pass's scene table is written by the kernel
that opens its chain of launches, while those after it are set up, so none of
them may hold an entry of the table before.  Images and gradients are those of
each batch alone in a workspace of its own."""
import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _item(seed, side, depth, levels):
    dev = torch.device("cuda:0")
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x, np.float32)).to(dev)  # noqa: E731
    V, F = S.icosphere(2 + seed % 2)
    V, F = t(V * (0.8 + 0.05 * seed)), torch.from_numpy(F).to(dev)
    cam = S.camera((0.3, 0.5 + 0.1 * seed, 3.0), (0.0, 0.0, 0.0), (0, 1, 0), 40.0, side, side)
    med = None
    if levels:
        # smooth values: a texture of unrelated entries makes the IoR gradient of a few rays dominate the sum
        res = [8 + 4 * l for l in range(levels)]
        g = torch.linspace(0.0, 1.0 + seed, 1 << 13, device=dev)
        table = torch.stack([g, 1.0 - 0.5 * g, 0.3 * g], 1)[None].repeat(levels, 1, 1) / levels
        med = dt.HashTexture(table.contiguous(), res, (-1.5,) * 3, (1.5,) * 3, 0.05 + 0.01 * seed)
    return dt.BatchItem(V, F, dt.build_bvh(V, F), dt.vertex_normals(V, F), torch.tensor([1.2 + 0.05 * seed], device=dev),
                        t([0.3, 0.1 * seed, 0.2]), t(S.sh_env_map(32, 16, seed)), t(cam.as_array()[None]), side, side,
                        dt.Params(depth), medium=med)


def _pass(items, ws, outs):
    _, tape = dt.render_batch(items, ws=ws, outs=outs, check=False)
    return dt.render_batch_backward(tape, outs)


@pytest.mark.parametrize("side", [24, 200])  # four lanes per ray; the persistent traversal in bucket order
def test_batches_back_to_back_in_one_workspace(side):
    # scenes, and levels of their hash textures (0: none)
    batches = [[(0, 0), (1, 0), (2, 0)], [(3, 3), (0, 0)], [(2, 1), (4, 5), (1, 0), (3, 2)], [(4, 2), (2, 4)], [(1, 0), (0, 0)]]
    batches = [[_item(s, side + 2 * s, 3 + s, l) for s, l in b] for b in batches]
    image = lambda it: torch.empty(1, it.height, it.width, 3, device="cuda")  # noqa: E731
    want, cap = [], 0
    for items in batches:
        ws = dt.Workspace(sum(it.n_primary for it in items) * 16, "cuda")
        cap = max(cap, ws.capacity)
        outs = [image(it) for it in items]
        grads = _pass(items, ws, outs)
        torch.cuda.synchronize()
        want.append((outs, grads))
    ws, got = dt.Workspace(cap, "cuda"), None
    for _ in range(4):
        got = []
        for items in batches:
            outs = [image(it) for it in items]
            got.append((outs, _pass(items, ws, outs)))
    torch.cuda.synchronize()
    for (outs, grads), (o2, g2) in zip(got, want):
        for x, y in zip([*outs, *sum(grads, ())], [*o2, *sum(g2, ())]):  # sums of the same terms in another order
            assert float((x - y).abs().max()) <= 1e-4 * float(y.abs().max()) + 1e-6
