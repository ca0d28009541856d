"""Warps of a partial tile that have no element of the launch read no face of it:
the tensor-core kernels' tile arithmetic (csrc/kernels.cuh) in a host program,
and the acoustic kernel on a fluid whose last tile leaves warps empty."""

import os
import shutil
import subprocess

import pytest

from _cases import make_pair, rel_l2, to_gpu_layout, to_oracle_layout

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2107_06640_gb300", "csrc")

HARNESS = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <vector>
#include "kernels.cuh"
using namespace adg;
// every face of the segment's elements by exactly one lane, and no other face
template <int TE, int EW>
int check(int64_t first, int64_t n, int S) {
  Seg s{};
  s.v_begin = first * S;
  s.n = n * S;
  const Segs g = make_segs(&s, 1, TE);
  std::vector<int> seen((first + n) * 4, 0);
  for (int64_t tl = 0; tl < g.first[g.n]; ++tl)
    for (int w = 0; w < TE / EW; ++w) {
      const TilePart p = tile_part<TE, EW>(g, tl, w);
      for (int lane = 0; lane < 32; ++lane) {
        const int64_t f = lane_face(p.v0, p.nE, lane, S);
        if (f < -1 || f >= (first + n) * 4) return 1;
        if (f >= 0) ++seen[f];
      }
    }
  for (int64_t f = 0; f < (first + n) * 4; ++f)
    if (seen[f] != (f >= first * 4 ? S : 0)) return 2;
  return 0;
}
int main() {
  for (int S : {1, 3})
    for (int64_t first : {0, 5})
      for (int64_t n = 1; n <= 70; ++n) {
        const int a = check<kTileElemsFluid, kRowElemsFluid>(first, n, S), b = check<kTileElems, kRowElems>(first, n, S);
        if (a || b) {
          std::printf("S %d, %lld elements from %lld: %d %d\n", S, (long long)n, (long long)first, a, b);
          return 1;
        }
      }
  std::printf("ok\n");
}
"""


def test_lane_faces_stay_within_the_segment(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_2107_06640_gb300 import build
    libdir = os.path.dirname(build.build())
    src, exe = str(tmp_path / "bounds.cpp"), str(tmp_path / "bounds")
    open(src, "w").write(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I" + CSRC, src, "-L" + libdir, "-ladg", "-Xlinker", "-rpath," + libdir, "-o",
                    exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("N", [4, 5])
def test_acoustic_tile_with_empty_warps_at_the_end_of_the_mesh(N):
    """No sea surface: the fluid is the last range of the library's order, 108 = 3 x 32 + 12 elements."""
    from synthetic.workloads import coupled_box, random_dofs
    m, mat = coupled_box(nxy=3, n_water=2, n_crust=1, L=6e3, depth=4e3, water=2e3)
    m.face_tag[m.face_tag == 2] = 1  # a free surface in the sea surface's place
    fluid = mat[2] == 0
    assert fluid.sum() % 32 in range(1, 25)
    o, s = make_pair(m, mat, N, precision=2, acoustic_ocean=True)
    Q0 = random_dofs((m.nt, s.B, 9), 19, N=N)
    Q0[fluid, :, 0:3] = Q0[fluid, :, 0:3].mean(axis=-1, keepdims=True)
    Q0[fluid, :, 3:6] = 0
    o.Q, o._D, o.t = Q0.copy(), None, 0.0
    s.set_dofs(to_gpu_layout(Q0))
    s.advance(2)
    for _ in range(2):
        o.advance_macro()
    assert rel_l2(to_oracle_layout(s.get_dofs()), o.Q) <= 2e-5  # the repository's parity tolerance of ADG_3XTF32
