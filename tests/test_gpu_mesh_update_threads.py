"""Two threads that update meshes of different size, each on its own stream:
the solver's launch takes a setting of the kernel (its shared memory), which
one thread must not change under the other.  Every update succeeds and gives
what the same updates give alone."""
import threading

import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _updates(V, F, grad, stream, steps):
    with torch.cuda.stream(stream):
        opt = dt.LargeStepsOptimizer(V, F, iters=1)
        for _ in range(steps):
            opt.step(grad)
        stream.synchronize()
    return V


def test_two_threads_update_meshes_of_different_size():
    dev = torch.device("cuda:0")
    meshes = []
    for level in (2, 6):
        V, F = S.icosphere(level)
        g = np.random.default_rng(level).normal(size=V.shape).astype(np.float32)
        meshes.append([torch.from_numpy(x).to(dev) for x in (V, F, g)])
    steps = 3000
    alone = [_updates(V.clone(), F, g, torch.cuda.Stream(dev), steps) for V, F, g in meshes]
    together, errors = [None, None], []

    def work(i):
        V, F, g = meshes[i]
        try:
            together[i] = _updates(V.clone(), F, g, torch.cuda.Stream(dev), steps)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append((i, repr(e)))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for a, b in zip(alone, together):
        assert torch.equal(a, b)
