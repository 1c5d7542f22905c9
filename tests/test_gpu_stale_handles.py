"""Handles that a pool has destroyed, because their job finished or failed, are refused by every call with
ICWF_ERR_ARG; none reads them."""
import ctypes as ct

import numpy as np
import pytest

from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")


def submit(pool, w, steps):
    sim = g.Icwf(g.params_from(w, precision=0), w.V)
    sim.init_from_density(w.psi0, 1)
    h = sim.release()
    return h, g.icwf_pool_submit(pool, h, steps)


def test_calls_with_a_destroyed_jobs_handle():
    w = shin_metiu(n_traj=8, svd_rel_cutoff=1e-8)
    pool = g.icwf_pool_create(1 << 34, 3)
    jobs = [submit(pool, w, n) for n in (1, 1 << 40, 1 << 40)]
    g.icwf_pool_tick(pool)                                  # the first job finishes
    g.LIB.icwf_set_regularisation(jobs[1][0], -0.5)         # the second meets a negative pivot
    g.icwf_pool_tick(pool)
    assert [g.icwf_pool_poll(pool, i, w.nx, w.nR)[0] for _, i in jobs] == [2, 3, 1]
    n, p = ct.c_size_t(), ct.c_void_p()
    obs, info = g.icwf_obs(), g.icwf_info()
    psi0 = np.ascontiguousarray(w.psi0, dtype=complex).view(float).ctypes.data_as(ct.POINTER(ct.c_double))
    for h, _ in jobs[:2]:
        calls = [g.LIB.icwf_step(h, 1), g.LIB.icwf_observables(h, ct.byref(obs)),
                 g.LIB.icwf_observables_static(h, ct.byref(obs)), g.LIB.icwf_get_info(h, ct.byref(info)),
                 g.LIB.icwf_get_state(h, None, None, None, None, None), g.LIB.icwf_get_matrices(h, None, None, None),
                 g.LIB.icwf_state_bytes(h, ct.byref(n)), g.LIB.icwf_work_bytes(h, ct.byref(n)),
                 g.LIB.icwf_get_stream(h, ct.byref(p)), g.LIB.icwf_set_regularisation(h, 1e-6),
                 g.LIB.icwf_set_projectors(h, 0, None), g.LIB.icwf_init_from_density(h, psi0, 0),
                 g.LIB.icwf_pool_submit(pool, h, 1, None), g.LIB.icwf_destroy(h)]
        assert calls == [g.ICWF_ERR_ARG] * len(calls)
    assert b"not a live handle" in g.LIB.icwf_last_error(jobs[0][0])
    assert g.icwf_observables(jobs[2][0], w.nx, w.nR)["norm"] > 0   # a live job is read as before
    g.icwf_pool_destroy(pool)
    assert g.LIB.icwf_destroy(jobs[2][0]) == g.ICWF_ERR_ARG
