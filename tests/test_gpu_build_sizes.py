"""The BVH build at the sizes where its parts meet: one task of the small
builder and less, the first large task, a chunk and several, several levels
of several chunks, one tile of the scan and more; repeated centroids that no
bin can split.  The closest hit does not depend on the tree, so the binned
SAH build and the LBVH find the same triangles at the same t, bit for bit,
and every ray aimed at a triangle's inside hits something no farther."""
import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nf", [1, 2, 3, 4, 5, 33, 127, 128, 129, 512, 513, 1024, 1025, 2047, 2050, 4096, 40000])
def test_build_sizes(nf):
    rng = np.random.default_rng(nf)
    c = rng.normal(size=(nf, 1, 3))
    if nf in (128, 513, 4096):  # many triangles about few centres: bins that cannot split, median splits
        c = c[rng.integers(0, 3, nf)]
    V = (c + rng.normal(scale=0.3 / nf ** (1 / 3), size=(nf, 3, 3))).astype(np.float32).reshape(-1, 3)
    F = np.arange(3 * nf, dtype=np.int32).reshape(nf, 3)
    o = rng.normal(size=(500, 3)) * 3.0
    k = rng.integers(0, nf, 500)
    w = 0.1 + 0.7 * rng.dirichlet((1.0, 1.0, 1.0), 500)  # well inside
    d = (V.reshape(nf, 3, 3)[k] * w[:, :, None]).sum(1) - o
    far = torch.from_numpy(np.linalg.norm(d, axis=1)).cuda()
    o, d = (torch.from_numpy(x.astype(np.float32)).cuda() for x in (o, d / np.linalg.norm(d, axis=1, keepdims=True)))
    Vt, Ft = torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda()
    got = []
    for builder in (0, 1):
        old = dt.set_tuning(bvh_builder=builder)
        try:
            got.append(dt.closest_hit(dt.build_bvh(Vt, Ft), o, d))
        finally:
            dt.set_tuning(**old)
    (tri0, tbb0), (tri1, tbb1) = got
    assert torch.equal(tri0, tri1) and torch.equal(tbb0, tbb1)
    assert (tri1 >= 0).all()
    # the aimed point's distance, up to the rounding of the aim (2^-24 of each coordinate, seen at grazing angles)
    assert (tbb1[:, 0].double() <= far + 1e-2).all()
