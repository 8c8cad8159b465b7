"""What a step brings into L2 ahead of its loads is what it will load: the node of each plane that
the prefetch names (kbc_device.cuh, compiled for the host) against the addressing of the step."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1507_02518_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
MAIN = r'''
#include <cstdio>
#include "kbc_device.cuh"
using namespace kbc;
template <int MODE> int check(uint32_t nx, uint32_t ny, uint32_t nz) {
  Geo g = {};
  g.nx = nx, g.ny = ny, g.nz = nz, g.nxy = nx * ny, g.P = (uint64_t)nx * ny * nz;
  int bad = 0;
  for (int i = 0; i < 27; ++i) {
    const int plane = MODE == MODE_AA_ODD ? 26 - i : i;
    const int sh = MODE == MODE_AA_EVEN ? 0 : -1;  // loads come from x + sh v_i
    if (plane != Pattern<MODE>::load_plane(i) || sh != Pattern<MODE>::load_shift) ++bad;
    const int vy = i / 3 % 3 - 1, vz = i / 9 - 1;
    for (uint64_t n = 0; n < g.P; ++n) {
      const uint64_t m = ahead_node<MODE>(g, plane, n);
      if (m >= g.P) ++bad;
      const int y = (int)(n / nx % ny), z = (int)(n / g.nxy);
      if (y == 0 || y + 1 == (int)ny) continue;
      const uint64_t zz = (uint64_t)((z + sh * vz + (int)nz) % (int)nz);
      if (m != n % nx + (uint64_t)(y + sh * vy) * nx + zz * g.nxy) ++bad;
    }
  }
  return bad;
}
int main() {
  int bad = 0;
  const uint32_t s[5][3] = {{3, 3, 3}, {8, 5, 4}, {7, 3, 9}, {64, 6, 3}, {5, 16, 7}};
  for (auto& b : s)
    bad += check<MODE_PULL>(b[0], b[1], b[2]) + check<MODE_AA_EVEN>(b[0], b[1], b[2]) +
           check<MODE_AA_ODD>(b[0], b[1], b[2]);
  printf("%d\n", bad);
  return bad != 0;
}
'''


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc is not here")
def test_prefetched_nodes_are_the_loaded_ones(tmp_path):
    (tmp_path / "m.cu").write_text(MAIN)
    exe = str(tmp_path / "m")
    subprocess.run([NVCC, "-std=c++17", "-I" + CSRC, "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", str(tmp_path / "m.cu"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
