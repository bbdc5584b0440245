"""The cell of a medium's sample, and the order in which samples are summed.
A sample is at ((o + s d) - lo) scale, rounded after the fused o + s d, the
difference and the product, in every pass: the gradient of a table of unrelated
entries jumps at a cell's faces, so a position formed in another order puts
samples near a face into another cell.  The optical depth is summed sample by
sample, level by level, however many lanes share a segment: the IoR gradient
near the critical angle is so ill-conditioned that another last bit of a depth
moves it by up to 5e-5.  The device functions are compiled by themselves and
compared, bit for bit, with the same operations on the host; cells also where a
segment is called inside its box (no clamping), on boxes up to 3000 of their
sides from the origin."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2603_00413_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cmath>
#include <vector>
#include "dt_medium.cuh"
using namespace dt;
struct Seg { float o[3], d[3], t, s, lo[3], scale[3]; int n; };
struct Cell { int i[3]; float f[3]; int inside; };
__global__ void k_cells(const Seg* seg, Cell* out, int count) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= count) return;
  const Seg S = seg[q];
  const MediumView g{nullptr, S.n, S.n, S.n, load3(S.lo), load3(S.scale), 0.01f, 0, nullptr};
  const Lattice T = lattice_of<false>(g, 0, load3(S.o), load3(S.d));
  const bool in = lattice_inside(T, S.t);
  const LatticeCell c = in ? lattice_cell<true>(T, S.s) : lattice_cell<false>(T, S.s);
  out[q] = Cell{{c.i, c.j, c.k}, {c.fx, c.fy, c.fz}, in};
}
__global__ void k_depths(const Seg* seg, MediumView g, float3* one, float3* four, int count) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x, w = q / 4;
  if (q < count) one[q] = medium_depth<true>(g, load3(seg[q].o), load3(seg[q].d), seg[q].t);
  const bool on = w < count;
  const Seg S = seg[on ? w : 0];
  const float3 sum = medium_depth_warp<true>(g, load3(S.o), load3(S.d), on ? S.t : 0.f, on);
  if (on && (q & 3) == 0) four[w] = sum;
}
// Depths of `count` segments through a dense grid of n^3 values (xyz of mu) over lo, scale of the first
// segment, or (levels > 0) a hash texture: bad[0] differ between four lanes and one, bad[1] (grid) from the host.
extern "C" int depths(const Seg* seg, int count, const float* mu, int entries, int n, float step, const GridLevel* lev,
                      int levels, int* bad) {
  Seg* ds = nullptr;
  float3* dd = nullptr;
  float4* dm = nullptr;
  GridLevel* dl = nullptr;
  std::vector<float3> got(2 * count);
  if (cudaMalloc(&ds, count * sizeof(Seg)) || cudaMalloc(&dd, 2 * count * sizeof(float3)) ||
      cudaMalloc(&dm, entries * sizeof(float4)) || cudaMalloc(&dl, 16 * sizeof(GridLevel)))
    return -1;
  cudaMemcpy(ds, seg, count * sizeof(Seg), cudaMemcpyHostToDevice);
  cudaMemcpy(dm, mu, entries * sizeof(float4), cudaMemcpyHostToDevice);
  if (levels) cudaMemcpy(dl, lev, levels * sizeof(GridLevel), cudaMemcpyHostToDevice);
  const float* L = seg[0].lo;
  const float* sc = seg[0].scale;
  const MediumView g{dm, n, n, n, mk(L[0], L[1], L[2]), mk(sc[0], sc[1], sc[2]), step, levels, dl};
  k_depths<<<(4 * count + 255) / 256, 256>>>(ds, g, dd, dd + count, count);
  const cudaError_t e = cudaMemcpy(got.data(), dd, 2 * count * sizeof(float3), cudaMemcpyDeviceToHost);
  cudaFree(ds);
  cudaFree(dd);
  cudaFree(dm);
  cudaFree(dl);
  if (e) return -1;
  bad[0] = bad[1] = 0;
  for (int q = 0; q < count; ++q) {
    const float3 x = got[q], y = got[count + q];
    bad[0] += !(x.x == y.x && x.y == y.y && x.z == y.z);
    if (levels) continue;
    const Seg& S = seg[q];
    const int m = (int)std::floor(S.t / step);
    const float mh = (float)m * step, rest = S.t - mh;
    float sum[3] = {0.f, 0.f, 0.f};
    for (int i = 0; i <= m; ++i) {
      const float s = i < m ? ((float)i + 0.5f) * step : std::fmaf(0.5f, rest, mh), w = i < m ? step : rest;
      int c[3];
      float f[3];
      for (int a = 0; a < 3; ++a) {
        const float y = std::fmaf(S.d[a], s, S.o[a]) - L[a];
        const float u = std::fmin(std::fmax(y * sc[a], 0.0f), (float)(n - 1));
        c[a] = std::min((int)u, n - 2);
        f[a] = u - (float)c[a];
      }
      for (int ch = 0; ch < 3; ++ch) {
        auto at = [&](int x, int y, int z) { return mu[4 * (((c[2] + z) * n + c[1] + y) * n + c[0] + x) + ch]; };
        auto lerp = [](float a, float b, float t) { const float d = b - a; return std::fmaf(d, t, a); };
        const float y0 = lerp(lerp(at(0, 0, 0), at(1, 0, 0), f[0]), lerp(at(0, 1, 0), at(1, 1, 0), f[0]), f[1]);
        const float y1 = lerp(lerp(at(0, 0, 1), at(1, 0, 1), f[0]), lerp(at(0, 1, 1), at(1, 1, 1), f[0]), f[1]);
        sum[ch] = std::fmaf(lerp(y0, y1, f[2]), w, sum[ch]);
      }
    }
    bad[1] += !(x.x == sum[0] && x.y == sum[1] && x.z == sum[2]);
  }
  return 0;
}
// seg: `count` segments; bad: samples whose cell or fraction differs; returns the segments found inside, or -1
extern "C" int check(const Seg* seg, int count, int* bad) {
  Seg* ds = nullptr;
  Cell* dc = nullptr;
  std::vector<Cell> got(count);
  if (cudaMalloc(&ds, count * sizeof(Seg)) || cudaMalloc(&dc, count * sizeof(Cell))) return -1;
  cudaMemcpy(ds, seg, count * sizeof(Seg), cudaMemcpyHostToDevice);
  k_cells<<<(count + 255) / 256, 256>>>(ds, dc, count);
  const cudaError_t e = cudaMemcpy(got.data(), dc, count * sizeof(Cell), cudaMemcpyDeviceToHost);
  cudaFree(ds);
  cudaFree(dc);
  if (e) return -1;
  int inside = 0;
  *bad = 0;
  for (int q = 0; q < count; ++q) {
    bool same = true;
    for (int a = 0; a < 3; ++a) {
      const float x = std::fmaf(seg[q].d[a], seg[q].s, seg[q].o[a]);
      const float y = x - seg[q].lo[a];
      float u = y * seg[q].scale[a];
      u = std::fmin(std::fmax(u, 0.0f), (float)(seg[q].n - 1));
      const int i = std::min((int)u, seg[q].n - 2);
      same &= got[q].i[a] == i && got[q].f[a] == u - (float)i;
    }
    *bad += !same;
    inside += got[q].inside;
  }
  return inside;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cells")
    (d / "cells.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-I", B.CSRC, "-shared", "-o", str(d / "cells.so"),
                    str(d / "cells.cu")], check=True)
    return ctypes.CDLL(str(d / "cells.so"))


def _segments(count, nodes, shift, reach, rng, half=1.25):
    seg = np.zeros(count, [("o", "f4", 3), ("d", "f4", 3), ("t", "f4"), ("s", "f4"), ("lo", "f4", 3),
                           ("scale", "f4", 3), ("n", "i4")])
    a, b = (shift + rng.uniform(-half * reach, half * reach, (count, 3)) for _ in range(2))
    t = np.linalg.norm(b - a, axis=1)
    seg["o"], seg["d"], seg["t"] = a, (b - a) / t[:, None], t
    seg["s"] = (seg["t"] * rng.uniform(0, 1, count)).astype(np.float32)
    seg["lo"], seg["n"] = np.float32(shift - half), nodes
    seg["scale"] = np.float32(nodes - 1) / (np.float32(shift + half) - np.float32(shift - half))
    return seg


@pytest.mark.parametrize("nodes,shift,reach", [(16, 0.0, 0.9), (128, 0.0, 0.9), (128, 0.0, 1.5), (64, 30.0, 0.98),
                                               (1024, 8000.0, 0.99)])
def test_a_sample_lies_in_the_cell_of_its_rounded_position(lib, nodes, shift, reach):
    count = 1 << 20
    seg = _segments(count, nodes, shift, reach, np.random.default_rng(nodes))
    bad = ctypes.c_int()
    inside = lib.check(ctypes.c_void_p(seg.ctypes.data), count, ctypes.byref(bad))
    assert bad.value == 0, f"{bad.value} of {count} samples in another cell"
    assert inside > 0  # the branch without clamping is reached


@pytest.mark.parametrize("levels,reach,step", [(0, 0.9, 0.0198), (0, 1.5, 0.3), (1, 0.9, 0.0098), (5, 1.5, 0.05)])
def test_depths_are_summed_sample_by_sample(lib, levels, reach, step):
    rng = np.random.default_rng(levels)
    count, nodes = 10007, 33
    seg = _segments(count, nodes, 0.0, reach, rng)
    seg["t"][:5] = [0.0, 1e-7, step, np.float32(step) * 4, 3.7]  # no full step, whole steps
    table = 1 << 12
    mu = rng.uniform(0, 1, (levels * table if levels else nodes ** 3, 4)).astype(np.float32)
    lev = np.zeros(16, [("n", "i4"), ("mask", "u4"), ("off", "u4"), ("s", "f4", 3), ("pad", "i4", 2)])
    for l in range(levels):
        n = 9 * (l + 1)
        lev[l]["n"], lev[l]["off"], lev[l]["mask"] = n, l * table, table - 1 if n ** 3 > table else 0
        lev[l]["s"] = np.float32(n - 1) / np.float32(2.5)
    bad = (ctypes.c_int * 2)()
    p = lambda a: ctypes.c_void_p(a.ctypes.data)  # noqa: E731
    assert lib.depths(p(seg), count, p(mu), len(mu), nodes, ctypes.c_float(step), p(lev), levels, bad) == 0
    assert list(bad) == [0, 0]
