"""Small renders are traced with four lanes per ray on the 4-wide nodes, larger
ones with a lane per ray on the coded binary nodes.  At the
sizes where the small path changes its shape (one ray, a warp's last rays, one
ray per warp and several, the last size it takes), alone and in a batch, both
find the same first hits at the same distances, and the same paths but for rays
through an edge, where either of the two triangles may be found."""
import numpy as np
import pytest

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S
from tests.gpu_util import GpuScene
from tests.test_gpu_batch import _items

pytestmark = pytest.mark.gpu

SMALL = 40960  # camera rays of the largest small render


def _scene(name, w, h, views=1):
    if name == "triangle":
        V, F = np.float32([[-1, -1, 0], [1, -1, 0], [0, 1, 0]]), np.int32([[0, 1, 2]])
    else:
        V, F = S.icosphere(3)
        if name == "two":
            V, F = np.concatenate([V, V * np.float32(0.4) + np.float32([0.9, 0.5, 0.8])]), np.concatenate([F, F + len(V)])
    cam = S.camera((0.31, 0.52, 3.03), (0.013, 0.007, 0.0), (0, 1, 0), 45.0, w, h)
    return GpuScene(V, F, 1.4, (0.3, 0.1, 0.2), S.sh_env_map(32, 16, 0), [cam] * views, w, h, 6)


def _sorted_segments(tape, n):
    """Those of the first n camera rays."""
    si, sf = dt.dump_segments(tape)
    first = si[:, 0] < n
    si, sf = si[first].cpu().numpy(), sf[first].cpu().numpy()
    order = np.lexsort((si[:, 1], si[:, 0]))
    return si[order], sf[order]


@pytest.mark.parametrize("name", ["ico", "two", "triangle"])
@pytest.mark.parametrize("w,h", [(1, 1), (3, 1), (9, 7), (64, 76), (71, 69), (202, 202), (203, 202)])
def test_small_render_finds_the_same_paths(name, w, h):
    img, tape = _scene(name, w, h).render()
    si, sf = _sorted_segments(tape, w * h)
    img2, tape2 = _scene(name, w, h, 1 + SMALL // (w * h)).render()
    si2, sf2 = _sorted_segments(tape2, w * h)
    a, b = si[:, 1] == 1, si2[:, 1] == 1
    assert a.sum() == b.sum() == w * h
    # the same first hits, at the same distance; of two triangles at one distance either
    assert np.array_equal(si[a, 2] >= 0, si2[b, 2] >= 0)
    assert np.array_equal(sf[a, 0], sf2[b, 0])
    # rays through an edge to the last bit are at most a few in a hundred thousand
    allowed = max(2, int(1e-4 * len(si)))
    keys, keys2 = ({tuple(r) for r in x[:, :3].tolist()} for x in (si, si2))
    assert len(keys ^ keys2) <= 8 * allowed
    # sums of at most 2^6 terms of order one, in another order
    assert int(((img[0] - img2[0]).abs().amax(-1) > 1e-4).sum()) <= allowed


def test_small_batch_equals_its_scenes():
    sizes = [("ico", 20, 13), ("triangle", 5, 4), ("two", 33, 17)]
    scenes = [_scene(*s) for s in sizes]
    alone = [gs.render()[0] for gs in scenes]
    imgs, _ = dt.render_batch(_items(scenes))
    for x, y in zip(alone, imgs):
        assert float((x - y).abs().max()) < 1e-5
