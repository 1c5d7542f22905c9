"""The coefficient solve where its parts change with the size.

Two levels (double-float, from 27 blocks on): the trailing updates are digit products on the tensor cores.
Its arithmetic is good to 2^-44 (see icwf.h), so the factorisation and the solves leave a residual of
2^-43 = 1.1e-13 of b; an update without its last digit or level would leave 2^-41 and more.

Above N = 2048 the triangular solves run as a block per CTA with flags in global memory, in both
arithmetics, and a restored state needs no neighbour products there: the bounds of the smaller sizes,
1e-9 and 1e-11."""
import numpy as np
import pytest

from oracle.icwf import Icwf as Oracle, Params
from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")


def residual(sim, w):
    st = sim.state()
    o = Oracle(Params(w.nx, w.nR, w.x_min, w.x_max, w.R_min, w.R_max, w.mass_x, w.mass_R, w.dt, w.n_traj,
                      w.svd_rel_cutoff, w.s_reg_eps), w.V)
    ost = o.init_from_positions(w.psi0, st["x"], st["R"])
    b = w.dx * w.dR * np.einsum("ia,ja,ij->a", ost.psi.conj(), ost.chi.conj(), w.psi0, optimize=True)
    r = (sim.matrices()["S"] + w.s_reg_eps * np.eye(w.n_traj)) @ st["C"] - b
    return np.linalg.norm(r) / np.linalg.norm(b)


@pytest.mark.parametrize("N", [833, 959, 1024, 1500, 2048])
def test_two_level_residual(N):
    w = shin_metiu(n_traj=N, svd_rel_cutoff=1e-8, s_reg_eps=1e-4 if N <= 1024 else 1e-3)
    sim = g.Icwf(g.params_from(w, precision=2), w.V)
    sim.init_from_density(w.psi0, 5)
    assert residual(sim, w) < 2.0 ** -43
    sim.close()


@pytest.mark.parametrize("precision,solve_fp64", [(0, 0), (2, 1), (2, 0)])
def test_above_the_cluster_solve(precision, solve_fp64):
    w = shin_metiu(n_traj=2049, svd_rel_cutoff=1e-8, s_reg_eps=1e-3)
    p = g.params_from(w, precision=precision, solve_fp64=solve_fp64)
    a = g.Icwf(p, w.V)
    a.init_from_density(w.psi0, 5)
    assert residual(a, w) < (1e-11 if precision == 0 or solve_fp64 else 1e-9)
    a.step(1)
    blob = a.save_state()
    a.step(1)
    c = g.Icwf(p, w.V)
    c.load_state(blob)
    c.step(1)
    assert np.array_equal(a.state(False)["C"], c.state(False)["C"])
    a.close()
    c.close()
