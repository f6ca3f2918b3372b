"""The level search's list of lattice points keeps within its capacity for every count that an accepted grid can reach: the
rule of the kernels, compiled for the host, at the counts where a 32-bit one changes sign or wraps."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_00947_gb300", "csrc")
MAIN = r"""
#include <initializer_list>
#include <type_traits>
#include "pplist.cuh"
int main() {
  using namespace mgar;
  // the count of a grid of 2^26 elements, all points in the bracket
  const long long total = 125LL << 26;
  for (int cap : {1, 4, 4096, 17373979, 1 << 26}) {
    const long long at[] = {0, cap - 1LL, cap, cap + 1LL, (1LL << 31) - 1, 1LL << 31, (1LL << 31) + cap, (1LL << 32) - 1,
                            1LL << 32, (1LL << 32) + cap - 1, total - 1, total};
    for (long long k : at) {
      const PpCount slot = (PpCount)k;
      if ((long long)slot != k) return 1;
      if (pp_listed(slot, cap) != (k < cap)) return 2;
      if (pp_complete(slot, cap) != (k <= cap)) return 3;
    }
  }
  return std::is_same<decltype(PpCtrl::nlist), PpCount>::value && sizeof(PpCount) == 8 && PpCount(-1) > 0 ? 0 : 4;
}
"""


def test_list_keeps_within_its_capacity(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "main.cpp"
    src.write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-x", "c++", str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
