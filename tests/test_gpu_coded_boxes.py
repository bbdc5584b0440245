"""The binary nodes' 16-bit box codes never cull a box the ray touches: on
scenes that stress the codes (far and very far cameras, rays inside box
planes, flat and scaled meshes, meshes away from the origin), and on a scene
with a part the grid cannot resolve, which takes the exact boxes, every
segment's hit is the one the 4-wide nodes' float boxes find, bit for bit.
Only where a ray meets an edge do the two differ (the axis-aligned box, whose
flat boxes end at the edge): there the float boxes may cull one of the two
triangles by rounding, and the coded ones find the nearer or, at the same
distance, the smaller triangle, as the tie rule asks."""
import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S
from tests.gpu_util import GpuScene, segments_by_key

pytestmark = pytest.mark.gpu

# renders of up to 40960 rays are traced on the 4-wide nodes at either setting: the frame many times over
VIEWS = 22


def _two_parts(small, scale):
    """A large icosphere, and a detailed one `scale` of its size beside it."""
    V, F = S.icosphere(2)
    v, f = S.icosphere(small)
    return np.concatenate([V, v * scale + np.float32([1.5, 0, 0])]).astype(np.float32), np.concatenate([F, f + len(V)])


def _case(name):
    V, F = S.icosphere(3)
    eye, at, fov = (0.3, 0.5, 3.0), (0.0, 0.0, 0.0), 45.0
    if name == "box":  # rays parallel to, and inside, the planes of the boxes
        V, F = S.box_grid(6)
        eye, fov = (0.0, 0.0, 3.0), 60.0
    elif name == "slab":
        V, F = S.box_grid(5, (1.0, 1e-3, 0.5))
        eye = (0.2, 1.0, 2.0)
    elif name == "far":
        eye, fov = (300.0, 500.0, 3000.0), 0.05
    elif name == "very_far":
        eye, fov = (0.0, 0.0, 1e5), 0.0015
    elif name == "large":
        V, eye = V * np.float32(1e5), (3e4, 5e4, 3e5)
    elif name == "small":
        V, eye = V * np.float32(1e-3), (3e-4, 5e-4, 3e-3)
    elif name == "shifted":
        V, eye, at = V + np.float32([100, -50, 30]), (100.3, -49.5, 33.0), (100.0, -50.0, 30.0)
    elif name == "triangle":
        V, F = np.float32([[-1, -1, 0], [1, -1, 0], [0, 1, 0]]), np.int32([[0, 1, 2]])
    elif name == "unresolved":
        V, F = _two_parts(4, 2e-5)
        eye, at, fov = (1.5, 0.0, 1e-4), (1.5, 0.0, 0.0), 40.0
    elif name == "two_scales":
        V, F = _two_parts(3, 1e-2)
        eye, at, fov = (1.5, 0.02, 0.05), (1.5, 0.0, 0.0), 45.0
    return V, F, S.camera(eye, at, (0, 1, 0), fov, 48, 40)


@pytest.mark.parametrize("builder", [0, 1])
@pytest.mark.parametrize("name", ["box", "slab", "far", "very_far", "large", "small", "shifted", "triangle",
                                  "unresolved", "two_scales"])
def test_coded_boxes_find_the_hits_of_float_boxes(name, builder):
    V, F, cam = _case(name)
    old = dt.get_tuning()
    try:
        dt.set_tuning(bvh_builder=builder)
        t_min = 1e-5 * float(np.abs(V - V.mean(0)).max())
        gs = GpuScene(V, F, 1.4, (0.3, 0.1, 0.2), S.sh_env_map(32, 16, 0), [cam] * VIEWS, 48, 40, 5, t_min=t_min)
        got = {}
        for width in (2, 4):
            dt.set_tuning(bvh_width=width)
            img, tape = gs.render()
            si, sf = dt.dump_segments(tape)
            first = si[:, 0] < 48 * 40
            si, sf = si[first].cpu().numpy(), sf[first].cpu().numpy()
            order = np.lexsort((si[:, 1], si[:, 0]))
            got[width] = (si[order], sf[order])
    finally:
        dt.set_tuning(**old)
    assert (got[2][0][:, 2] >= 0).any()
    if name != "box":
        assert segments_by_key(got[2][0]) == segments_by_key(got[4][0])
        assert np.array_equal(got[2][1], got[4][1])
    # segments of the same ray in both trees: never a later hit, or a larger triangle at the same t
    row4 = {(int(r[0]), int(r[1])): k for k, r in enumerate(got[4][0])}
    same = 0
    for k, r in enumerate(got[2][0]):
        j = row4.get((int(r[0]), int(r[1])))
        if j is None or not np.array_equal(got[2][1][k, 3:9], got[4][1][j, 3:9]):
            continue
        t2, t4 = (float(f[0]) if i[2] >= 0 else np.inf for i, f in ((r, got[2][1][k]), (got[4][0][j], got[4][1][j])))
        assert t2 < t4 or (t2 == t4 and r[2] <= got[4][0][j][2]), (r, got[4][0][j], t2, t4)
        same += 1
    assert same >= 0.5 * len(got[2][0])
    # arbitrary rays take the same nodes: the rays of the tape, asked again
    o, d = (torch.from_numpy(np.ascontiguousarray(got[2][1][:, k:k + 3])).cuda() for k in (3, 6))
    cam_rays = got[2][0][:, 1] == 1
    tri, tbb = dt.closest_hit(gs.bvh, o[cam_rays].contiguous(), d[cam_rays].contiguous(), t_min=t_min)
    assert np.array_equal(tri.cpu().numpy(), got[2][0][cam_rays, 2])
    assert np.array_equal(tbb.cpu().numpy(), got[2][1][cam_rays, :3])
