"""A traversal order that is not one of its level is reported, by every
traversal alike: the lookup they share, compiled for the host."""
import subprocess

from paper_2603_00413_gb300 import build as B

SOURCE = r"""
#include "dt_internal.cuh"
#include <cstdio>
int main() {
  const uint32_t order[6] = {2, 0, 1, 3, 4, 0xffffffffu};
  uint32_t pos = 0;
  int bad = 0;
  for (uint32_t i = 0; i < 3; ++i) bad += !dt::order_position(order, i, 3, pos) || pos != order[i];
  for (uint32_t i = 3; i < 6; ++i) bad += dt::order_position(order, i, 3, pos);
  for (uint32_t i = 0; i < 3; ++i) bad += !dt::order_position(nullptr, i, 3, pos) || pos != i;
  std::printf("%d", bad);
}
"""


def test_an_entry_outside_the_level_is_reported(tmp_path):
    src, exe = tmp_path / "order.cu", tmp_path / "order"
    src.write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-I", B.CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "0"
    # the traversals (a lane per ray, four lanes per ray) read the order through it alone
    trace = open(B.CSRC + "/dt_trace.cu").read()
    assert trace.count("order_position(") >= 2 and "W.sflag[start + " not in trace and "order[" not in trace
