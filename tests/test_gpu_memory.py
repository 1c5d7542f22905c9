"""Device memory: a handle's device_bytes, by which pools admit it, are no more than what the library
before the sliced Grams reported (commit 2029912, recorded on a GB300), so whatever fitted a budget
still does; the work space beyond them is bounded by the batches of the FP64 mode's terms.

Bounds of the work space, by hand, in MB.  FP64, N = 16, 64 terms of at most eight digits: 12.6 of operands
(32 rows of 12 slices, 49 kB per digit of a term), 2.1 of Grams, 1.3 of bras and term sums: 16.  FP64 above:
a batch of 134 (128 MiB), bras of 32 bytes per point, Grams of the overlap and term sums of 16 N^2
bytes each or less, products of 6.1 kB per trajectory: 26 more at N = 256, 90 at 1024, 66 at 2049 on 64 x
64.  Mixed modes: the products, and nothing else."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

g = pytest.importorskip("paper_1805_11169_gb300")

# precision, solve_fp64, N, nx, nR, cutoff: rank, device_bytes then, work space in MB (FP64)
SHAPES = [((0, 0, 16, 128, 64, 0.0), 64, 825856, 16), ((0, 0, 256, 512, 256, 1e-12), 101, 15019008, 160),
          ((0, 0, 1024, 1024, 512, 1e-12), 155, 160979968, 224), ((2, 0, 64, 256, 128, 1e-8), 52, 22825216, 0),
          ((2, 0, 16, 64, 64, 1e-8), 23, 1002496, 0), ((2, 0, 333, 512, 128, 1e-8), 95, 348983808, 0),
          ((2, 1, 500, 512, 256, 1e-8), 96, 641934080, 0), ((1, 0, 512, 512, 256, 1e-8), 96, 656091904, 0),
          ((2, 0, 2049, 64, 64, 1e-8), 23, 583813888, 0), ((0, 0, 2049, 64, 64, 1e-8), 23, 486716672, 200)]


def make(precision, solve_fp64, N, nx, nR, cutoff):
    x, R = (np.arange(nx) + 0.5) / nx * 100 - 50, (np.arange(nR) + 0.5) / nR * 18 - 9
    p = g.icwf_params(nx=nx, nR=nR, x_min=-50.0, x_max=50.0, R_min=-9.0, R_max=9.0, mass_x=1.0, mass_R=1836.0,
                      dt=0.05, n_traj=N, precision=precision, svd_rel_cutoff=cutoff, s_reg_eps=1e-3, coeff_scheme=0,
                      max_rank=0, solve_fp64=solve_fp64, overlap_split=0)
    return g.Icwf(p, 1 / np.sqrt((x[:, None] - R[None]) ** 2 + 1.0)), x, R


@pytest.mark.parametrize("shape,rank,then,work", SHAPES)
def test_no_larger_than_before(shape, rank, then, work):
    sim, _, _ = make(*shape)
    info = sim.info()
    assert info["rank"] == rank and info["device_bytes"] <= then
    # (mixed modes: the last block padded to 32 trajectories, and the plan's tables)
    assert g.icwf_work_bytes(sim.h) <= (work * 1e6 if work else 6.2e3 * (shape[2] + 31) + 65536)
    sim.close()


def test_pool_with_the_budget_of_before():
    sim, x, R = make(*SHAPES[0][0])
    psi0 = np.exp(-0.1 * x[:, None] ** 2 - 0.5 * R[None] ** 2).astype(complex)
    sim.init_from_density(psi0 / np.sqrt(100 / 128 * 18 / 64 * np.sum(np.abs(psi0) ** 2)), 1)
    pool = g.icwf_pool_create(SHAPES[0][2], 1)
    job = g.icwf_pool_submit(pool, sim.release(), 2)
    for _ in range(2):
        g.icwf_pool_tick(pool)
    assert g.icwf_pool_poll(pool, job, 128, 64)[0] == 2
    g.icwf_pool_destroy(pool)
