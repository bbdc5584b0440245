"""The smallest renders (a few pixels: one ray, a warp's last rays) are, segment by
segment and bit for bit, those of the same frame traced with a lane per ray: no
allowance, since none of their rays meets an edge."""
import numpy as np
import pytest

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S
from tests.gpu_util import GpuScene

pytestmark = pytest.mark.gpu

SMALL = 40960  # camera rays of the largest small render


def _segments(gs, n):
    img, tape = gs.render()
    si, sf = dt.dump_segments(tape)
    first = si[:, 0] < n
    si, sf = si[first].cpu().numpy(), sf[first].cpu().numpy()
    order = np.lexsort((si[:, 1], si[:, 0]))
    return img[0].cpu().numpy(), si[order], sf[order]


@pytest.mark.parametrize("w,h", [(1, 1), (2, 1), (3, 1), (1, 5), (7, 3), (9, 7), (13, 11), (31, 1), (33, 5)])
@pytest.mark.parametrize("mesh", ["tori", "two", "grid"])
def test_a_few_pixels_are_the_same(mesh, w, h):
    if mesh == "tori":
        V, F = S.two_tori_mesh(24)
    elif mesh == "grid":  # no vertex or edge on an axis
        V, F = S.box_grid(5)
        a, b = np.float32(0.37), np.float32(0.81)
        R = np.float32([[np.cos(a), -np.sin(a), 0], [np.sin(a), np.cos(a), 0], [0, 0, 1]])
        V = V @ R @ np.float32([[1, 0, 0], [0, np.cos(b), -np.sin(b)], [0, np.sin(b), np.cos(b)]])
    else:
        V, F = S.icosphere(3)
        V, F = np.concatenate([V, V * np.float32(0.4) + np.float32([0.9, 0.5, 0.8])]), np.concatenate([F, F + len(V)])
    cam = S.camera((0.313, 0.527, 3.031), (0.0131, 0.0073, 0.0), (0, 1, 0), 41.0, w, h)
    env = S.sh_env_map(32, 16, 0)
    one, many = (GpuScene(V, F, 1.4, (0.3, 0.1, 0.2), env, [cam] * n, w, h, 6) for n in (1, 1 + SMALL // (w * h)))
    img, si, sf = _segments(one, w * h)
    img2, si2, sf2 = _segments(many, w * h)
    assert np.array_equal(si, si2) and np.array_equal(sf, sf2)
    # sums of at most 2^6 terms of order one, in another order
    np.testing.assert_allclose(img, img2, rtol=0, atol=2 ** 6 * 2 ** -23)
