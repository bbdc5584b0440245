"""The paper losses around the size from which four pixels share a thread, at every
remainder of the four, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2603_00413_gb300 as dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [65535, 65536, 65537, 65538, 65539])
def test_paper_loss_around_the_line(n):
    rng = np.random.default_rng(n)
    a, b = rng.uniform(0.05, 1.5, size=(2, n, 3)).astype(np.float32)
    g, loss = dt.paper_loss_grad(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), 0.6, 1.4)
    total, lc, lt, gref = O.paper_losses(a.astype(np.float64)[None], b.astype(np.float64)[None], 0.6, 1.4)
    # sums of 65,536 terms of one sign in 32 bits, by threads, warps and CTAs; gradients of a dozen operations
    np.testing.assert_allclose(loss.cpu().numpy(), [total, lc, lt], rtol=2e-5, atol=2e-6)
    np.testing.assert_allclose(g.cpu().numpy(), gref[0], rtol=2e-5, atol=1e-6 * np.abs(gref).max())
