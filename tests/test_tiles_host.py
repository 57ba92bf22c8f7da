"""The rule that chooses the backprojector's tiles (sipo_tiles.h) depends on the
shape alone, as the tiles enter the order of the sums: it compiles with the host
compiler, without CUDA or a device, and gives the choices of a part with 152 SMs at
the sizes beside the rule and on both sides of its limits."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_08997_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include "sipo_tiles.h"
int main() {
  const double counts[] = {1, 41, 134, 164, 227, 228, 286, 490};
  for (double n : counts) std::printf("%d ", sipo::bp_rows(n));
  // tiles of 8 rows; twice as many with half the rows
  const double eights[] = {1, 100, 122, 199, 200, 398, 399, 797, 798, 5000};
  for (double n : eights) {
    const sipo::BpPlan p = sipo::bp_split(180, [&](int rows) { return n * 8 / rows; });
    std::printf("%d:%d ", p.rows, p.split);
  }
  const int views[] = {1, 8, 13, 14, 27, 28, 55, 56, 60, 400};
  for (int k : views) std::printf("%d ", sipo::bp_split(k, [](int) { return 1.0; }).split);
  return 0;
}
"""


def test_tiles_follow_from_the_shape_alone(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "tiles.cpp", tmp_path / "tiles"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out[:8] == ["2", "2", "2", "2", "2", "8", "8", "8"]
    # shared until there are 1.75 * 3 * 152 = 798 tiles, by eight warps at most
    assert out[8:18] == ["1:3", "1:3", "1:3", "1:3", "2:2", "2:2", "4:1", "4:1", "8:0", "8:0"]
    # seven views a warp at least
    assert out[18:] == ["0", "0", "0", "1", "1", "2", "2", "3", "3", "3"]


def test_the_solver_asks_no_device_for_them():
    text = open(os.path.join(CSRC, "sipo_abi.cu")).read()
    body = text[text.index("void choose_bp_tiles()"):text.index("void setup(")]
    assert "device_sms" not in body
