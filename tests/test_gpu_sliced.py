"""Matrix elements and the reconstruction by sliced Grams (csrc/k_sliced.cu) at the sizes where their
tiling changes: trajectories around the 32/64/128 unit widths and the 128-row tiles, grids below
one K slice (8 points), at several accumulation chunks (4096 points) and in between, full and
truncated rank, both operand-piece types and the split-product overlap.

Oracle: its formulas in FP64 on the GPU's own CWFs and positions.  Bounds: the FP64 mode's digits
resolve 2^-56 of a column's largest component, below the oracle's own FP64 sums (n 2^-53 = 4.5e-13
at 4096 points): 1e-12.  Mixed modes: S is the Gram of 24-bit fixed-point CWFs (1e-7; 22-bit digits
on 4096 points: 1e-6), Heff and the split-product overlap carry the pieces' rounding (1e-5); the
reconstruction in 5 digits resolves 2^-34 of the largest term (1e-7 of the densities)."""
import numpy as np
import pytest

from oracle.icwf import Icwf as Oracle, Params
from workloads import shin_metiu_potential

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")

CASES = [(1, 8, 8, 0, 0.0, 0), (16, 128, 64, 0, 0.0, 0), (31, 16, 8, 0, 0.0, 0), (33, 64, 32, 0, 1e-12, 0),
         (64, 4096, 16, 0, 1e-12, 0), (65, 2048, 64, 0, 1e-12, 0), (130, 256, 16, 0, 1e-12, 0),
         (257, 512, 64, 0, 1e-12, 0), (16, 64, 64, 2, 1e-8, 0), (32, 64, 128, 1, 1e-8, 0), (65, 256, 64, 2, 0.0, 0),
         (128, 128, 64, 2, 1e-8, 0), (129, 256, 64, 1, 1e-8, 0), (300, 1024, 64, 2, 1e-8, 0),
         (40, 4096, 64, 2, 1e-8, 0), (129, 256, 64, 2, 1e-8, 1), (50, 2048, 64, 1, 1e-8, 1)]


@pytest.mark.parametrize("N,nx,nR,mode,cutoff,split", CASES)
def test_matrices_and_densities(N, nx, nR, mode, cutoff, split):
    rng = np.random.default_rng(N)
    dx, dR = 40.0 / nx, 14.0 / nR
    x, R = -20.0 + (np.arange(nx) + 0.5) * dx, -7.0 + (np.arange(nR) + 0.5) * dR
    V = shin_metiu_potential(x, R)
    psi0 = np.exp(-0.1 * (x[:, None] - 0.5) ** 2 - 0.3 * (R[None, :] + 2) ** 2 + 0.2j * x[:, None] * R[None, :])
    psi0 /= np.sqrt(dx * dR * np.sum(np.abs(psi0) ** 2))
    p = g.icwf_params(nx=nx, nR=nR, x_min=-20.0, x_max=20.0, R_min=-7.0, R_max=7.0, mass_x=1.0, mass_R=1836.0,
                      dt=0.05, n_traj=N, precision=mode, svd_rel_cutoff=cutoff, s_reg_eps=1e-3, coeff_scheme=0,
                      max_rank=0, solve_fp64=0, overlap_split=split)
    sim = g.Icwf(p, V)
    sim.init_from_positions(psi0, rng.uniform(-4, 4, N), rng.uniform(-4, 1, N))
    sim.step(1)
    st, m, obs = sim.state(), sim.matrices(), sim.observables()
    sim.close()
    o = Oracle(Params(nx, nR, -20.0, 20.0, -7.0, 7.0, 1.0, 1836.0, 0.05, N, cutoff, 1e-3), V)
    S = o.overlaps(st["psi"], st["chi"])[2]
    H = o.heff_factorised(st["psi"], st["chi"], st["x"], st["R"])
    dens = np.abs((st["psi"] * st["C"]) @ st["chi"].T) ** 2

    def rel(a, b):
        return np.linalg.norm(a - b) / np.linalg.norm(b)

    tol_s = 1e-12 if mode == 0 else (1e-5 if split else (1e-7 if nx <= 2048 else 1e-6))
    assert rel(m["S"], S) < tol_s
    assert np.array_equal(m["S"], m["S"].conj().T)
    assert rel(m["Heff"], H) < (1e-12 if mode == 0 else 1e-5)
    tol = 1e-12 if mode == 0 else 1e-7
    assert rel(obs["rho_x"], dR * dens.sum(axis=1)) < tol and rel(obs["rho_R"], dx * dens.sum(axis=0)) < tol
