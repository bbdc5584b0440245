"""The refit at the sizes where its parts meet: less than a CTA's leaves, one
leaf more, several CTAs whose nodes are shared.  A tree refitted to moved
vertices, by either builder, finds the hits of the tree built for them, bit for
bit: both hold boxes that contain their triangles, and the closest hit depends
on nothing else."""
import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("builder", [0, 1])
@pytest.mark.parametrize("nf", [1, 2, 3, 511, 512, 513, 514, 1024, 1025, 5000, 30011])
def test_refit_equals_build(nf, builder):
    rng = np.random.default_rng(nf)
    V = (rng.normal(size=(nf, 1, 3)) + rng.normal(scale=0.3 / nf ** (1 / 3), size=(nf, 3, 3))).astype(np.float32)
    W = (V + rng.normal(scale=0.1, size=(nf, 1, 3))).astype(np.float32)
    F = torch.arange(3 * nf, dtype=torch.int32).reshape(nf, 3).cuda()
    Vt, Wt = (torch.from_numpy(x.reshape(-1, 3)).cuda() for x in (V, W))
    o = torch.from_numpy((rng.normal(size=(4000, 3)) * 3.0).astype(np.float32)).cuda()
    d = torch.from_numpy(W.mean(1)[rng.integers(0, nf, 4000)]).cuda() - o
    d = d / d.norm(dim=1, keepdim=True)
    old = dt.set_tuning(bvh_builder=builder)
    try:
        fresh, moved = dt.build_bvh(Wt, F), dt.build_bvh(Vt, F)
        dt.refit_bvh(moved, Wt, F)
        want = dt.closest_hit(fresh, o, d)
        got = dt.closest_hit(moved, o, d)
        assert (want[0] >= 0).any()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        dt.refit_bvh(moved, Vt, F)  # and back
        got, want = dt.closest_hit(moved, o, d), dt.closest_hit(dt.build_bvh(Vt, F), o, d)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    finally:
        dt.set_tuning(**old)
