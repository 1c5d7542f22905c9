"""The double-float triangular solves at the edges of their 32-row blocks and of the cluster's 16 CTAs:
one block (no neighbour products), two and three (no second neighbour; every block among the first three
rows), a ragged last block, 16 / 17 blocks (the CTAs' second round), and a restored state, whose
neighbour products are recomputed from the saved factor.

Bound of the residual, fixed beforehand: 2^-44 per operation, N <= 545 terms per entry and the explicit
inverses of 32 x 32 diagonal blocks with condition numbers up to 1 / eps = 1e4 give 545 * 6e-14 * 1e4 =
3e-7 at the very worst; rounding errors of random sign stay far below, and the bar is the 1e-9 of the
other sizes' test."""
import numpy as np
import pytest

from oracle.icwf import Icwf as Oracle, Params
from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")

EPS = 1e-4


@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 64, 65, 96, 97, 129, 511, 512, 513, 545])
def test_residual_and_restored_state(N):
    w = shin_metiu(n_traj=N, svd_rel_cutoff=1e-8, s_reg_eps=EPS)
    a = g.Icwf(g.params_from(w, precision=2), w.V)
    a.init_from_density(w.psi0, 5)
    st = a.state()
    o = Oracle(Params(w.nx, w.nR, w.x_min, w.x_max, w.R_min, w.R_max, w.mass_x, w.mass_R, w.dt, w.n_traj,
                      w.svd_rel_cutoff, EPS), w.V)
    ost = o.init_from_positions(w.psi0, st["x"], st["R"])
    b = w.dx * w.dR * np.einsum("ia,ja,ij->a", ost.psi.conj(), ost.chi.conj(), w.psi0, optimize=True)
    r = (a.matrices()["S"] + EPS * np.eye(N)) @ st["C"] - b
    assert np.linalg.norm(r) / np.linalg.norm(b) < 1e-9
    a.step(2)
    blob = a.save_state()
    a.step(2)
    c = g.Icwf(g.params_from(w, precision=2), w.V)
    c.load_state(blob)
    c.step(2)
    assert np.array_equal(a.state()["C"], c.state()["C"])
    a.close()
    c.close()
