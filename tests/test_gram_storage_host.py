"""Host test of the Hermitian Grams' storage (sliced.cuh, Tri, compiled as plain C++): for every ensemble
size the units of 32, 64 and 128 kets cover every ket of every upper-triangle tile once and no tile
beyond it, their stores stay apart and inside size(), and every element k_heff reads is stored."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1805_11169_gb300", "csrc")

PROG = r'''
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "sliced.cuh"
using namespace icwf::sl;
int main(int argc, char** argv) {
  for (int a = 1; a < argc; ++a)
    for (int t = 32; t <= 128; t *= 2) {
      const int N = atoi(argv[a]);
      const Tri tri(N);
      std::vector<char> seen(tri.size(), 0);
      for (int v = 0; v < tri.units(t); ++v) {
        int tile, part, I, J;
        tri.unit(v, t, tile, part);
        tri_tile(tile, I, J);
        if (tile >= tri.tiles() || J >= tri.T || part * t >= N - J * MT) return printf("N %d unit %d: beyond\n", N, v), 1;
        const int nc = (tile < tri.full ? MT : tri.kl) - part * t;
        for (int k = 0; k < t && k < nc; ++k)
          for (int b = 0; b < tri.br; ++b) {
            const size_t at = tri.at(tile) + ((size_t)part * t + k) * tri.br + b;
            if (at >= tri.size() || seen[at]++) return printf("N %d unit %d: store %zu\n", N, v, at), 1;
          }
      }
      for (int tile = 0; tile < tri.tiles(); ++tile) {
        int I, J;
        tri_tile(tile, I, J);
        for (int p = 0; p < 16; ++p) {   // k_heff's patches
          const int ac = (p & 3) * 32, bc = (p >> 2) * 32;
          if (I * MT + ac >= N || J * MT + bc >= N) continue;
          for (int b = bc; b < bc + 32; ++b)
            for (int c = ac; c < ac + 32; ++c)
              if (!seen[tri.at(tile) + (size_t)b * tri.br + c]) return printf("N %d tile %d: hole\n", N, tile), 1;
        }
      }
    }
  return 0;
}
'''


def test_units_cover_the_stored_tiles(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "p.cpp").write_text(PROG)
    subprocess.run([cxx, "-O2", "-std=c++17", "-w", "-I", CSRC, str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")],
                   check=True)
    sizes = list(range(1, 300)) + [383, 384, 385, 416, 700, 1023, 1024, 1025, 2049]
    r = subprocess.run([str(tmp_path / "p")] + [str(n) for n in sizes], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
