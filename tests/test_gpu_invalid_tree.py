"""A tree that failed its validation is left alone by a refit (its leaves may never
have been set), and rays are refused by it."""
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_refit_leaves_an_invalid_tree_alone():
    V, F = S.icosphere(3)
    V, F = torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda()
    bvh = dt.build_bvh(V, F)
    bvh.buf[12:16].view(torch.int32).fill_(1)  # BvhHeader::corrupt
    before = bvh.buf.clone()
    dt.refit_bvh(bvh, V * 2.0, F)
    assert torch.equal(bvh.buf, before)
    tri, _ = dt.closest_hit(bvh, torch.zeros(4, 3, device="cuda"), torch.ones(4, 3, device="cuda"))
    assert (tri == -2).all()  # and so do rays
