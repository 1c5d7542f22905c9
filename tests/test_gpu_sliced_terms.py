"""FP64 matrix elements when the rank-k terms are of very different shape, and when there are more of
them than one batch of Grams holds.

A term that sits on a few grid points is worth more there than its singular value says: its digits are
chosen by its largest value.  Reference: the oracle's formulas on the GPU's own CWFs.  Bound for the
local term: library and oracle take their factors from different SVDs, each off by 2^-53 of the largest
singular value s_1, so Heff agrees to 2^-53 s_1 / |Heff|.  Bound for many terms: the 1e-12 of the
other FP64 matrix elements."""
import numpy as np
import pytest

from oracle.icwf import Icwf as Oracle, Params
from workloads import shin_metiu_potential

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")


def matrices(V, nx, nR, psi0, xs, Rs, dt):
    p = g.icwf_params(nx=nx, nR=nR, x_min=-20.0, x_max=20.0, R_min=-7.0, R_max=7.0, mass_x=1.0, mass_R=1836.0,
                      dt=dt, n_traj=len(xs), precision=0, svd_rel_cutoff=0.0, s_reg_eps=1e-3, coeff_scheme=0,
                      max_rank=0, solve_fp64=0, overlap_split=0)
    sim = g.Icwf(p, V)
    sim.init_from_positions(psi0, xs, Rs)
    sim.step(1)
    st, m, rank = sim.state(), sim.matrices(), sim.info()["rank"]
    sim.close()
    o = Oracle(Params(nx, nR, -20.0, 20.0, -7.0, 7.0, 1.0, 1836.0, dt, len(xs), 0.0, 1e-3), V)
    return (m["S"], o.overlaps(st["psi"], st["chi"])[2], m["Heff"],
            o.heff_factorised(st["psi"], st["chi"], st["x"], st["R"]), rank)


def grid(nx, nR):
    dx, dR = 40.0 / nx, 14.0 / nR
    return -20.0 + (np.arange(nx) + 0.5) * dx, -7.0 + (np.arange(nR) + 0.5) * dR, dx, dR


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_narrow_feature_beside_a_large_smooth_one():
    nx, nR = 256, 64
    x, R, dx, dR = grid(nx, nR)
    far = 1000.0 * np.exp(-0.5 * ((x[:, None] - 12) / 3) ** 2 - 0.5 * (R[None, :] - 4) ** 2)
    V = far + np.exp(-2 * (x[:, None] / dx) ** 2 - 2 * (R[None, :] / dR) ** 2)
    psi0 = np.exp(-(x[:, None] / (4 * dx)) ** 2 - (R[None, :] / (4 * dR)) ** 2 + 0.2j * x[:, None] * R[None, :])
    psi0 /= np.sqrt(dx * dR * np.sum(np.abs(psi0) ** 2))
    rng = np.random.default_rng(24)
    S, So, H, Ho, _ = matrices(V, nx, nR, psi0, rng.uniform(-2, 2, 24) * dx, rng.uniform(-2, 2, 24) * dR, 1e-3)
    centred = V - V.mean(1)[:, None] - V.mean(0)[None, :] + V.mean()
    assert rel(S, So) < 1e-12
    assert np.linalg.norm(H - Ho) < 2.0 ** -53 * np.linalg.svd(centred, compute_uv=False)[0]


@pytest.mark.parametrize("N", [20, 129])
def test_more_terms_than_a_batch_of_grams(N):
    nx, nR = 256, 256
    x, R, dx, dR = grid(nx, nR)
    psi0 = np.exp(-0.1 * (x[:, None] - 0.5) ** 2 - 0.3 * (R[None, :] + 2) ** 2 + 0.2j * x[:, None] * R[None, :])
    psi0 /= np.sqrt(dx * dR * np.sum(np.abs(psi0) ** 2))
    rng = np.random.default_rng(N)
    S, So, H, Ho, rank = matrices(shin_metiu_potential(x, R), nx, nR, psi0, rng.uniform(-4, 4, N),
                                  rng.uniform(-4, 1, N), 0.05)
    assert rank > 125
    assert rel(S, So) < 1e-12 and rel(H, Ho) < 1e-12
