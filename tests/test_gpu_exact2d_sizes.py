"""The exact propagator's register FFT passes at every length they are compiled for (8 .. 4096, each with
its own split into passes), in both directions, against numpy's fft2 in the oracle.

Bound, fixed beforehand: FP64 rounding of 3 steps x 4 transforms x 12 stages, a few 2^-53 each and
random in sign, stays below 1e-13 of the largest component; the bar is 1e-12."""
from types import SimpleNamespace

import numpy as np
import pytest

from oracle.exact2d import Exact2D as OracleExact2D
from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")


@pytest.mark.parametrize("nx,nR", [(8, 4096), (16, 2048), (32, 1024), (64, 512), (128, 256), (256, 128), (512, 64),
                                   (1024, 32), (2048, 16), (4096, 8), (8, 8)])
def test_every_length(nx, nR):
    w = SimpleNamespace(**vars(shin_metiu()))
    w.nx, w.nR = nx, nR
    rng = np.random.default_rng(nx + nR)
    w.V = rng.standard_normal((nx, nR))
    psi = rng.standard_normal((nx, nR)) + 1j * rng.standard_normal((nx, nR))
    o = OracleExact2D(nx, nR, w.x_min, w.x_max, w.R_min, w.R_max, w.mass_x, w.mass_R, w.dt, w.V)
    ref = o.run(psi, 3)
    e = g.Exact2D(g.params_from(w), w.V)
    e.set_state(psi)
    e.step(2)
    e.step(1)
    out = e.state()
    assert np.max(np.abs(out - ref)) / np.max(np.abs(ref)) < 1e-12
    e.step(0)
    assert np.array_equal(e.state(), out)
    e.close()
