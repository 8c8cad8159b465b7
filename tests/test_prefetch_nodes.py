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
// the largest boxes: nodes near 2^31
template <int MODE> int check_large(uint32_t nx, uint32_t ny, uint32_t nz) {
  Geo g = {};
  g.nx = nx, g.ny = ny, g.nz = nz, g.nxy = nx * ny, g.P = (uint64_t)nx * ny * nz;
  int bad = 0;
  for (uint32_t plane = 0; plane < 27; ++plane)
    for (uint64_t k = 0; k < g.P; k += g.P / 1000 - 1) {
      const int64_t o = ((int)(plane / 3 % 3) - 1) * (int64_t)nx + ((int)(plane / 9) - 1) * (int64_t)g.nxy;
      for (uint64_t n : {k, g.P - 1 - k}) {
        int64_t m = (int64_t)n + (MODE == MODE_PULL ? -o : MODE == MODE_AA_ODD ? o : 0);
        m = (m + (int64_t)g.P) % (int64_t)g.P;
        bad += ahead_node<MODE>(g, plane, (uint32_t)n) != (uint64_t)m;
      }
    }
  return bad;
}
int main() {
  int bad = 0;
  const uint32_t l[3][3] = {{1290, 1290, 1290}, {26754, 26754, 3}, {3, 3, 238609294}};
  for (auto& b : l)
    bad += check_large<MODE_PULL>(b[0], b[1], b[2]) + check_large<MODE_AA_EVEN>(b[0], b[1], b[2]) +
           check_large<MODE_AA_ODD>(b[0], b[1], b[2]);
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
