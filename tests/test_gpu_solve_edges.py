"""The cluster's triangular solves, double-float and FP64, at the edges of their 32-row blocks and of the
16 warps: one block (no neighbour products), two and three (every block among the first three rows), a
ragged last block, 16 / 17 and 32 / 33 blocks (a warp's second and third block), 64 (the largest), and a
restored state, whose neighbour products are recomputed from the saved factor.  From 27 blocks on the
double-float factorisation behind them has tensor-core trailing updates (832: the last single launch,
833 and 959: ragged trailing matrices after the first panel, 2048: ten panels).

Bounds of the residual, fixed beforehand.  Double-float: 2^-44 per operation, N <= 545 terms per entry and
the explicit inverses of 32 x 32 diagonal blocks with condition numbers up to 1 / eps = 1e4 give 545 *
6e-14 * 1e4 = 3e-7 at the very worst; rounding errors of random sign stay far below, and the bar is the
1e-9 of the other sizes' test.  FP64: 2^-53 instead, 1e-11 as there."""
import numpy as np
import pytest

from oracle.icwf import Icwf as Oracle, Params
from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")

EPS = 1e-4


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 64, 65, 96, 97, 129, 511, 512, 513, 545, 832, 833, 959, 1024, 1025, 2048])
def test_residual_and_restored_state(N, fp64):
    w = shin_metiu(n_traj=N, svd_rel_cutoff=1e-8, s_reg_eps=EPS if N <= 1024 else 1e-3)
    eps = w.s_reg_eps
    a = g.Icwf(g.params_from(w, precision=2, solve_fp64=fp64), w.V)
    a.init_from_density(w.psi0, 5)
    st = a.state()
    o = Oracle(Params(w.nx, w.nR, w.x_min, w.x_max, w.R_min, w.R_max, w.mass_x, w.mass_R, w.dt, w.n_traj,
                      w.svd_rel_cutoff, eps), w.V)
    ost = o.init_from_positions(w.psi0, st["x"], st["R"])
    b = w.dx * w.dR * np.einsum("ia,ja,ij->a", ost.psi.conj(), ost.chi.conj(), w.psi0, optimize=True)
    r = (a.matrices()["S"] + eps * np.eye(N)) @ st["C"] - b
    assert np.linalg.norm(r) / np.linalg.norm(b) < (1e-11 if fp64 else 1e-9)
    a.step(2)
    blob = a.save_state()
    a.step(2)
    c = g.Icwf(g.params_from(w, precision=2, solve_fp64=fp64), w.V)
    c.load_state(blob)
    c.step(2)
    assert np.array_equal(a.state()["C"], c.state()["C"])
    a.close()
    c.close()
