"""Builds and mesh updates on a stream that has a few of the device's SMs (a green
context): the cooperative grids shrink until they fit, and the results are those
on the whole device."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S

pytestmark = pytest.mark.gpu

RESOURCE_BYTES = 256  # of CUdevResource (144) and room to spare
SM = 1                # CU_DEV_RESOURCE_TYPE_SM, CU_GREEN_CTX_DEFAULT_STREAM, CU_STREAM_NON_BLOCKING


@pytest.fixture()
def few_sms():
    """A stream of a green context with at least 8 SMs, and their number."""
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    for name in ("cuDeviceGetDevResource", "cuDevSmResourceSplitByCount", "cuDevResourceGenerateDesc", "cuGreenCtxCreate",
                 "cuGreenCtxStreamCreate"):
        if not hasattr(cu, name):
            pytest.skip(f"the driver has no {name}")

    def call(f, *a):
        r = f(*a)
        if r:
            pytest.skip(f"{f.__name__}: CUDA error {r}")

    whole, part, rest = (ctypes.create_string_buffer(RESOURCE_BYTES) for _ in range(3))
    dev, groups = ctypes.c_int(), ctypes.c_uint(1)
    desc, ctx, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    call(cu.cuDeviceGet, ctypes.byref(dev), 0)
    call(cu.cuDeviceGetDevResource, dev, whole, SM)
    call(cu.cuDevSmResourceSplitByCount, part, ctypes.byref(groups), whole, rest, 0, 8)
    call(cu.cuDevResourceGenerateDesc, ctypes.byref(desc), part, 1)
    call(cu.cuGreenCtxCreate, ctypes.byref(ctx), desc, dev, SM)
    call(cu.cuGreenCtxStreamCreate, ctypes.byref(stream), ctx, SM, 0)
    yield torch.cuda.ExternalStream(stream.value), int.from_bytes(part.raw[96:100], "little")
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


def _mesh(level):
    V, F = S.icosphere(level)
    V = V * (1.0 + 0.1 * np.sin(7.0 * V[:, :1]))
    return torch.from_numpy(V.astype(np.float32)).cuda(), torch.from_numpy(F).cuda()


def test_mesh_update_on_a_few_sms(few_sms):
    stream, sms = few_sms
    assert 8 <= sms < 64
    V, F = _mesh(5 if sms < 20 else 6)  # one CTA per 512 vertices: more than the SMs
    assert V.shape[0] > 512 * sms
    g = torch.sin(4.0 * V)
    want = dt.LargeStepsOptimizer(V.clone(), F).step(g).clone()
    torch.cuda.synchronize()
    opt = dt.LargeStepsOptimizer(V.clone(), F)
    torch.cuda.synchronize()
    got = opt.step(g, stream=stream)
    torch.cuda.synchronize()
    # other partial sums: the solver's residual tolerance on vertices of order one
    assert torch.isfinite(got).all() and float((got - want).abs().max()) < 1e-5


def test_build_on_a_few_sms(few_sms):
    stream, sms = few_sms
    V, F = _mesh(6)  # 81,920 triangles, a CTA for 512 each, three per SM
    assert F.shape[0] > 512 * 3 * sms
    o = torch.randn(20000, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(0)) * 3.0
    d = -o / o.norm(dim=1, keepdim=True)
    want = dt.closest_hit(dt.build_bvh(V, F), o, d)
    bvh = dt.Bvh(F.shape[0], V.device)
    torch.cuda.synchronize()
    bvh.build(V, F, stream=stream)
    got = dt.closest_hit(bvh, o, d, stream=stream)
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
