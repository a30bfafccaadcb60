"""Co-resident CTAs of kernels that hold tensor memory: 512 columns per SM bound them, whatever
registers and shared memory would allow."""
import os
import re
import shutil
import subprocess

from paper_2604_17109_gb300 import build as pkg_build

MAIN = """
#include <cstdio>
#include "kernels.h"
int main() {
  const int cases[][3] = {{1, 512, 1}, {2, 512, 1}, {3, 512, 1}, {2, 256, 2}, {3, 256, 2}, {4, 128, 4}, {1, 64, 1}, {0, 512, 0}};
  int bad = 0;
  for (const auto& c : cases) bad += pim::resident_ctas(c[0], c[1]) != c[2];
  return bad;
}
"""


def test_tensor_memory_bounds_the_ctas_of_an_sm(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(pkg_build._nvcc()))), "include")
    cxx = shutil.which("g++") or shutil.which("c++")
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-I", pkg_build.CSRC, "-I", cuda, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_every_count_of_resident_blocks_goes_through_it():
    """Each use of the occupancy call in a kernel file that allocates tensor memory is bounded."""
    for name in ("k_sweep_big.cu", "k_sweep_mid.cu"):
        text = open(os.path.join(pkg_build.CSRC, name)).read()
        assert "tmem_alloc(" in text
        assert len(re.findall(r"cudaOccupancyMaxActiveBlocksPerMultiprocessor\(", text)) == len(
            re.findall(r"resident_ctas\(per_sm, ", text))
