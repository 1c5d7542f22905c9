"""Host test of the double-float trailing update's numbers (sliced.cuh: fixed_of_f32, cut_digits, compiled as
plain C++): the seven digits of a pair hi + lo, and the products kept.  CPU only.

Bounds.  A pair below 2^e is rounded twice to units of 2^(e - 48), half a unit each.  Of a product the pairs of
digits (p, q) with p + q < 7 are kept, which weigh 2^-(12 + 7 (p + q)) and are at most 2^12: of those dropped
at most 6 2^-49 + 5 2^-56 + ... < 2^-46.4 is lost per product of values below 1, and the roundings add 2^-47."""
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
int main() {
  float h, l;
  int e;
  while (scanf("%a %a %d", &h, &l, &e) == 3) {
    const int q = 48 - e;
    int d[7];
    cut_digits<7>(fixed_of_f32(h, q) + fixed_of_f32(l, q), d);
    for (int v : d) printf("%d ", v);
    printf("\n");
  }
}
'''


@pytest.fixture(scope="module")
def digits(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("pairs")
    (d / "p.cpp").write_text(PROG)
    subprocess.run([cxx, "-O1", "-std=c++17", "-w", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)

    def run(pairs, e):
        text = "".join("%s %s %d\n" % (float(h).hex(), float(l).hex(), e) for h, l in pairs)
        out = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True).stdout
        return [[int(t) for t in line.split()] for line in out.splitlines()]

    return run


def pairs_of(rng, n, spread):
    x = rng.uniform(-1, 1, n) * 2.0 ** -rng.integers(0, spread + 1, n)
    h = x.astype(np.float32)
    return list(zip(h, (x - h).astype(np.float32)))


@pytest.mark.parametrize("e,spread", [(0, 0), (0, 60), (-100, 20), (90, 3)])
def test_digits_of_a_pair(digits, e, spread):
    rng = np.random.default_rng(spread)
    s = np.float32(2.0 ** e)
    pairs = [(h * s, l * s) for h, l in pairs_of(rng, 300, spread)]
    pairs += [(s * np.float32(1 - 2.0 ** -24), s * np.float32(2.0 ** -25)), (np.float32(0), np.float32(0)), (-s * np.float32(0.5), s * np.float32(2.0 ** -49))]
    for (h, l), dg in zip(pairs, digits(pairs, e)):
        assert abs(dg[0]) <= 64 and all(-64 <= t <= 63 for t in dg[1:])
        v = sum(Fraction(t, 2 ** (6 + 7 * p)) for p, t in enumerate(dg)) * Fraction(2) ** e
        assert abs(v - Fraction(float(h)) - Fraction(float(l))) <= Fraction(2) ** (e - 48)


@pytest.mark.parametrize("spread", [0, 30])
def test_kept_products(digits, spread):
    rng = np.random.default_rng(7 + spread)
    x, y = pairs_of(rng, 128, spread), pairs_of(rng, 128, spread)
    err = Fraction(0)
    for (h, l), (a, b), p, q in zip(x, y, digits(x, 0), digits(y, 0)):
        exact = (Fraction(float(h)) + Fraction(float(l))) * (Fraction(float(a)) + Fraction(float(b)))
        kept = sum(Fraction(p[i] * q[j], 2 ** (12 + 7 * (i + j))) for i in range(7) for j in range(7 - i))
        assert abs(kept - exact) < Fraction(3, 2 ** 47)
        err += kept - exact
    assert abs(err) < 128 * Fraction(3, 2 ** 47)
