"""A CWF with a NaN (put into a saved state): the step reports ICWF_ERR_NUMERIC, S is NaN in the rows and
columns of the trajectories whose CWFs are, and nowhere else (in the FP64 mode Heff too), the densities
are NaN, and a good state loaded into the handle afterwards runs as before."""
import numpy as np
import pytest

from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")


@pytest.mark.parametrize("precision,N,a", [(0, 20, 5), (0, 150, 149), (2, 20, 5), (2, 150, 149), (1, 40, 33)])
def test_nan_stays_with_its_trajectory(precision, N, a):
    w = shin_metiu(n_traj=N, svd_rel_cutoff=1e-8, s_reg_eps=1e-4)
    sim = g.Icwf(g.params_from(w, precision=precision), w.V)
    sim.init_from_density(w.psi0, 2)
    good = sim.save_state()
    column = np.ascontiguousarray(sim.state()["psi"][:, a]).astype(np.complex128 if precision == 0 else np.complex64)
    at = good.find(column.tobytes())
    assert at >= 0
    column[w.nx // 3] = np.nan
    sim.load_state(good[:at] + column.tobytes() + good[at + column.nbytes:])
    with pytest.raises(g.IcwfError) as e:
        sim.step(1)
    assert e.value.status == g.ICWF_ERR_NUMERIC
    m, st = sim.matrices(), sim.state()
    bad = ~np.isfinite(st["psi"]).all(axis=0) | ~np.isfinite(st["chi"]).all(axis=0)
    assert bad[a] and bad.sum() < N // 2
    for q in (m["S"], m["Heff"]) if precision == 0 else (m["S"],):
        assert np.array_equal(np.isnan(q.real), bad[:, None] | bad[None, :])
    assert np.isnan(sim.observables()["rho_x"]).any()
    sim.load_state(good)
    sim.step(2)
    fresh = g.Icwf(g.params_from(w, precision=precision), w.V)
    fresh.init_from_density(w.psi0, 2)
    fresh.step(2)
    assert np.array_equal(sim.state()["C"], fresh.state()["C"])
    sim.close()
    fresh.close()
