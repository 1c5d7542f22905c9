"""Host unit test of the sliced Grams' number formats and index arithmetic
(paper_1805_11169_gb300/csrc/sliced.cuh, compiled as plain C++): digits of FP64 numbers, 64-bit
integer sums back to FP64, the operand swizzle and the triangular tile index.  CPU only."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1805_11169_gb300", "csrc")

PROG = r'''
#include <cstdio>
#include "sliced.cuh"
using namespace icwf::sl;
template <int D> void digits(double x, int q) { int d[D]; digits_of<D>(x, q, d); for (int v : d) printf("%d ", v); printf("\n"); }
int main() {
  char t; 
  while (scanf(" %c", &t) == 1) {
    if (t == 'd') { double x; int q, D; scanf("%la %d %d", &x, &q, &D);
      printf("%d ", exponent_above_f64(abs_bits(x)));
      if (D == 2) digits<2>(x, q); else if (D == 3) digits<3>(x, q); else if (D == 5) digits<5>(x, q); else digits<8>(x, q); }
    if (t == 'f') { long long v; int sh; scanf("%lld %d", &v, &sh); printf("%a\n", fixed_to_f64(v, sh)); }
    if (t == 's') { int d; scanf("%d", &d); printf("%a\n", (double)small_int_to_float(d)); }
    if (t == 'w') { int r, p; scanf("%d %d", &r, &p); printf("%d\n", swizzle32(r, p)); }
    if (t == 't') { int n, I, J; scanf("%d", &n); tri_tile(n, I, J); printf("%d %d\n", I, J); }
  }
}
'''


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("sliced")
    (d / "p.cpp").write_text(PROG)
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-w", "-I", CSRC, str(d / "p.cpp"), "-o",
                    str(d / "p")], check=True)
    return lambda text: subprocess.run([str(d / "p")], input=text, capture_output=True, text=True,
                                       check=True).stdout.split("\n")[:-1]


@pytest.mark.parametrize("D", [2, 3, 5, 8])
def test_digits_represent_the_number_to_the_last_digit(prog, D):
    rng = np.random.default_rng(D)
    xs = np.concatenate([rng.uniform(-1, 1, 200) * 10.0 ** rng.integers(-300, 300, 200),
                         [1.0, -1.0, np.nextafter(1.0, 0), -np.nextafter(2.0, 0), 0.0, 5e-324, 1e-310]])
    e = [int(np.frexp(x)[1]) if x else 0 for x in xs]
    out = prog("".join("d %s %d %d\n" % (float(x).hex(), 6 + 7 * (D - 1) - k, D) for x, k in zip(xs, e)))
    for x, k, line in zip(xs, e, out):
        v = [int(t) for t in line.split()]
        if x:
            assert abs(Fraction(x)) < Fraction(2) ** v[0] and abs(Fraction(x)) >= Fraction(2) ** (v[0] - 1)
            assert v[0] == k
        dg = v[1:]
        assert abs(dg[0]) <= 64 and all(-64 <= t <= 63 for t in dg[1:])
        s = sum(Fraction(t, 2 ** (6 + 7 * p)) for p, t in enumerate(dg)) * Fraction(2) ** k
        assert abs(s - Fraction(x)) <= Fraction(2) ** (k - 6 - 7 * (D - 1) - 1)


def test_integer_sums_convert_with_one_rounding(prog):
    rng = np.random.default_rng(1)
    vs = [int(t) for t in rng.integers(-2 ** 62, 2 ** 62, 300)] + [0, 1, -1, 2 ** 62, -2 ** 62, 2 ** 53 + 1]
    vs += [int(t) >> int(s) for t, s in zip(vs[:200], rng.integers(0, 62, 200))]
    sh = [int(t) for t in rng.integers(-200, 100, len(vs))]
    for v, s, line in zip(vs, sh, prog("".join("f %d %d\n" % t for t in zip(vs, sh)))):
        got, want = Fraction(float.fromhex(line)), Fraction(v) * Fraction(2) ** s
        assert abs(got - want) <= abs(want) * Fraction(1, 2 ** 53)


def test_small_integers_and_indices(prog):
    assert [float.fromhex(t) for t in prog("".join("s %d\n" % d for d in range(-130, 131)))] == list(range(-130, 131))
    at = [int(t) for t in prog("".join("w %d %d\n" % (r, p) for r in range(128) for p in (0, 1)))]
    # every 16-byte half of the tile once, rows in place, address bit 4 XORed with address bit 7
    assert sorted(at) == list(range(0, 128 * 32, 16))
    for i, a in enumerate(at):
        r, p = i // 2, i % 2
        assert a // 32 == r and ((a >> 4) & 1) == p ^ ((r * 32 >> 7) & 1)
    n = 8256   # all tiles of 128 row blocks (16384 trajectories)
    ij = [tuple(int(v) for v in t.split()) for t in prog("".join("t %d\n" % k for k in range(n)))]
    assert ij == [(i, j) for j in range(128) for i in range(j + 1)]
