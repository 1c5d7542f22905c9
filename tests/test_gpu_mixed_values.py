"""The mixed modes' numbers stay those their users have: values recorded on a GB300 from the library as of
commit 2029912 (tests/golden/mixed_heff.npz, mixed_cwf.npz).

Heff's rounding is part of a mixed mode's results: (S + eps I)^-1 with eps = 1e-6 amplifies it, so
another rounding of the products, a more exact one too, moves the densities by 2e-5 within a few steps.
Bounds: Heff at t = 0 from the same complex64 CWFs and the same sums, one FP32 rounding, 2^-24 = 6e-8;
the densities after 10 steps (0.5 a.u.) the agreement of FP32 results, 2e-5."""
import os

import numpy as np
import pytest

from workloads import shin_metiu

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")

GOLDEN = os.path.join(os.path.dirname(__file__), "golden")
X_RANGE = {256: (-60.0, 60.0), 512: (-60.0, 60.0)}


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def start(n, nx, mode, eps):
    w = shin_metiu(nx=nx, x_range=X_RANGE[nx], nR=128, R_range=(-9.0, 9.0), n_traj=n, dt=0.05, svd_rel_cutoff=1e-8,
                   s_reg_eps=eps)
    sim = g.Icwf(g.params_from(w, precision=mode), w.V)
    sim.init_from_density(w.psi0, 3)
    return sim


@pytest.mark.parametrize("key,n,nx,mode,eps", [("heff_tf32", 717, 512, g.ICWF_MIXED_TF32X3, 1e-6),
                                               ("heff_bf16", 300, 256, g.ICWF_MIXED_BF16X3, 1e-4)])
def test_heff_of_the_initial_state(key, n, nx, mode, eps):
    sim = start(n, nx, mode, eps)
    want = np.load(os.path.join(GOLDEN, "mixed_heff.npz"))[key]
    assert rel(sim.matrices()["Heff"][:24, :24], want) < 6e-8
    sim.close()


def test_densities_after_ten_steps():
    sim = start(717, 512, g.ICWF_MIXED_TF32X3, 1e-6)
    sim.step(10)
    obs = sim.observables()
    want = np.load(os.path.join(GOLDEN, "mixed_heff.npz"))
    assert rel(obs["rho_x"], want["rho_x"]) < 2e-5 and rel(obs["rho_R"], want["rho_R"]) < 2e-5
    sim.close()


def test_cwfs_after_one_step():
    """The propagator's FP32 tables are rounded to nearest: the same CWFs to a unit of FP32, 2^-25 = 3e-8 in
    the 2-norm (tables rounded to the nearest modulus instead: 1.9e-7)."""
    sim = start(717, 512, g.ICWF_MIXED_TF32X3, 1e-6)
    sim.step(1)
    want = np.load(os.path.join(GOLDEN, "mixed_cwf.npz"))["psi"]
    assert rel(sim.state()["psi"][:, :2], want) < 3e-8
    sim.close()
