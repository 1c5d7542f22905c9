"""What the framework is measured on: ICWF time stepping through the public binding, from the
smallest serving job to the largest ensembles, in the arithmetic modes a user chooses between, the
exact 2D propagation the method is compared with, and the serving pool.

A pass is what a user's program repeats: advance the handle by a few steps, read the observables
and the trajectories.  FP64 handles return FP64 numbers.  The mixed modes carry their CWFs in
complex64, and a program keeps what it reads from them in that precision, so their results are
returned in FP32.  The small cases return the CWFs too (a program that keeps every step).  The
coefficients C are not returned: they are fixed only up to the near-null space of S (two FP64
solvers differ there by 1e-8, two mixed ones by 1e-1), which the wavefunction, and with it the
densities, populations, energy and trajectories, does not see.
"""
import math

import numpy as np
import torch

import paper_1805_11169_gb300 as icwf
from workloads.models import cavity_potential, cell_grid, shin_metiu_potential, soft_coulomb

MODES = {"fp64": icwf.ICWF_FP64, "bf16x3": icwf.ICWF_MIXED_BF16X3, "tf32x3": icwf.ICWF_MIXED_TF32X3}
N_STATES = 3
# half-widths of the x grids, by model and number of points
X_HALF = {"shin_metiu": {128: 50.0, 256: 60.0, 512: 60.0, 1024: 100.0},
          "cavity": {256: 40.0, 512: 60.0, 1024: 60.0, 2048: 80.0}}
R_HALF = {"shin_metiu": {64: 9.0, 128: 9.0, 256: 9.0, 512: 9.5},
          "cavity": {64: 15.0, 128: 20.0, 256: 30.0}}
PROTON = 1836.0


def _icwf(name, model, nx, nR, n, mode, steps, **over):
    c = dict(name=name, kind="icwf", model=model, nx=nx, nR=nR, n=n, mode=mode, steps=steps,
             dt=0.05 if model == "shin_metiu" else 0.01,
             cutoff=1e-12 if mode == "fp64" else 1e-8,
             eps=1e-6 if model == "shin_metiu" and mode != "bf16x3" else 1e-4,
             frozen=False, solve_fp64=False, cwfs=False)
    c.update(over)
    return c


def listed():
    return [
        # the smallest job a user runs, one step at a time: FP64, 16 trajectories, full rank
        _icwf("fp64_tiny", "shin_metiu", 128, 64, 16, "fp64", 1, cutoff=0.0,
              cwfs=True),
        # the smallest job of the serving stream
        _icwf("mixed_small_job", "shin_metiu", 256, 128, 64, "tf32x3", 2, cwfs=True),
        # an ordinary job with a ragged ensemble, matrices frozen over the step (one factorisation;
        # it wants the larger eps)
        _icwf("mixed_ragged_frozen", "shin_metiu", 512, 128, 333, "tf32x3", 2, frozen=True, eps=1e-4),
        # an ordinary job in the faster split-BF16 mode, at the eps that mode wants
        _icwf("mixed_bf16_job", "shin_metiu", 512, 256, 512, "bf16x3", 2),
        # mixed assembly with the FP64 solver, for the users who want FP64 residuals
        _icwf("mixed_solve_fp64", "shin_metiu", 512, 256, 500, "tf32x3", 2, solve_fp64=True),
        # the paper's proton-coupled electron transfer at its own scale (the headline workload)
        _icwf("mixed_paper", "shin_metiu", 1024, 512, 1024, "tf32x3", 2),
        # the paper's cavity application at its own scale
        _icwf("mixed_cavity", "cavity", 2048, 256, 1024, "tf32x3", 2),
        # the largest ensemble of the serving stream on the paper's grid
        _icwf("mixed_large", "shin_metiu", 1024, 512, 2048, "tf32x3", 1),
        # FP64 at an ensemble that accuracy studies use
        _icwf("fp64_study", "shin_metiu", 512, 256, 256, "fp64", 2),
        # FP64 at the headline size: the reference the mixed modes are judged against
        _icwf("fp64_paper", "shin_metiu", 1024, 512, 1024, "fp64", 1),
        # the exact 2D solution of the same problem, advanced to the next comparison point
        dict(name="exact2d_paper", kind="exact2d", model="shin_metiu", nx=1024, nR=512, steps=50,
             dt=0.05),
        # the serving pool: four live jobs of different sizes and models, two ticks
        dict(name="pool_ticks", kind="pool", jobs="sm256x128x64,cav512x128x128,sm512x128x200,sm256x128x384",
             steps=2),
    ]


def draw(rng):
    """Any of the three kinds; ensembles spread over the logarithm of 16..2048 (16..700 in FP64),
    odd sizes included."""
    kind = rng.choice(["icwf"] * 8 + ["exact2d", "pool"])
    if kind == "exact2d":
        nx, nR = rng.choice([(128, 64), (256, 128), (512, 128), (512, 256), (1024, 512)])
        return dict(kind="exact2d", model="shin_metiu", nx=nx, nR=nR, steps=rng.randrange(5, 41),
                    dt=rng.choice([0.02, 0.05, 0.1]))
    if kind == "pool":
        jobs = []
        for _ in range(rng.randrange(2, 5)):
            model = rng.choice(["sm", "sm", "cav"])
            nx, nR = rng.choice([(256, 128), (512, 128)]) if model == "sm" else (512, 128)
            lo = 40 if model == "sm" else 100
            jobs.append("%s%dx%dx%d" % (model, nx, nR, round(math.exp(rng.uniform(math.log(lo), math.log(500))))))
        return dict(kind="pool", jobs=",".join(jobs), steps=rng.randrange(1, 4))
    mode = rng.choice(["tf32x3", "tf32x3", "tf32x3", "bf16x3", "fp64"])
    model = rng.choice(["shin_metiu", "shin_metiu", "cavity"])
    grids = {"shin_metiu": [(128, 64), (256, 128), (512, 128), (512, 256), (1024, 512)],
             "cavity": [(256, 64), (512, 128), (1024, 128), (2048, 256)]}[model]
    # the cavity is stiff in small ensembles run for long
    lo, hi = 16 if model == "shin_metiu" else 128, 700 if mode == "fp64" else 2048
    n = round(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    nx, nR = rng.choice(grids)
    c = _icwf("", model, nx, nR, n, mode, rng.randrange(1, 3), frozen=rng.random() < 0.15,
              solve_fp64=mode != "fp64" and rng.random() < 0.15, cwfs=n < 100)
    if c["frozen"]:
        c["eps"] = 1e-4
    c.pop("name")
    return c


# ---- the problem: potential, initial state, projectors, positions ------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _states(V, x, half, n):
    """The lowest n electronic states of T_x + V(., R_j) for every j, real, normalised with dx, in
    the sine basis of the box |x| < half (their tails are below 1e-6 there); continuous in R.
    V: nx x nR.  Returns n x nR x nx."""
    nb, dx = 56, x[1] - x[0]
    inside = np.abs(x) < half
    k = np.arange(1, nb + 1) * math.pi / (2.0 * half)
    s = np.zeros((len(x), nb))
    s[inside] = np.sin((x[inside, None] + half) * k[None, :]) / math.sqrt(half)
    s, k = torch.as_tensor(s, device=_device()), torch.as_tensor(k, device=_device())
    H = torch.matmul(s.T * dx, torch.as_tensor(V.T.copy(), device=s.device)[:, :, None] * s)
    H = H + torch.diag(0.5 * k * k)
    c = torch.linalg.eigh(H)[1][:, :, :n]                           # nR x nb x n
    flip = torch.sign((c[1:] * c[:-1]).sum(1))
    c = torch.cat([c[:1], c[1:] * torch.cumprod(flip, 0)[:, None, :]])
    phi = torch.matmul(s, c).permute(2, 0, 1)                       # n x nR x nx
    lead = phi[:, 0, :].gather(1, phi[:, 0, :].abs().argmax(1, keepdim=True))
    phi = phi * torch.sign(lead)[:, :, None]
    return (phi / torch.sqrt(dx * (phi * phi).sum(2, keepdim=True))).cpu().numpy()


def _problem(c, seed):
    """Grids, masses, V, Psi0, projectors and sampled positions, from the seed alone."""
    rng = np.random.RandomState(seed)
    hx, hR = X_HALF[c["model"]][c["nx"]], R_HALF[c["model"]][c["nR"]]
    x, dx = cell_grid(c["nx"], -hx, hx)
    R, dR = cell_grid(c["nR"], -hR, hR)
    if c["model"] == "shin_metiu":
        V = shin_metiu_potential(x, R, Rf=rng.uniform(4.6, 5.4))
        phi = _states(V, x, 32.0, N_STATES)
        g = np.exp(-(R - rng.uniform(-4.3, -3.7)) ** 2 * (0.5 * 2.85))
        psi0, mass_R = phi[1].T * g[None, :], PROTON
    else:
        lam, omega = rng.uniform(0.3, 0.6), 0.3945
        V = cavity_potential(x, R, omega, lam)
        phi = _states(V, x, 32.0, N_STATES)
        atom = _states(soft_coulomb(x)[:, None], x, 32.0, 2)[1, 0]
        psi0, mass_R = np.outer(atom, np.exp(-0.5 * omega * R * R)), 1.0
    psi0 = (psi0 / math.sqrt(dx * dR * float(np.sum(psi0 ** 2)))).astype(np.complex128)
    w = dict(nx=c["nx"], nR=c["nR"], x_min=-hx, x_max=hx, R_min=-hR, R_max=hR, mass_x=1.0,
             mass_R=mass_R, dt=c["dt"], V=V, psi0=psi0, phi=np.ascontiguousarray(phi),
             x=x, R=R, dx=dx, dR=dR)
    if "n" in c:
        cum = np.cumsum((psi0.real ** 2).ravel())
        cell = np.minimum(np.searchsorted(cum, rng.uniform(size=c["n"]) * cum[-1], side="right"), cum.size - 1)
        w["xs"] = x[cell // c["nR"]] + rng.uniform(-0.5, 0.5, c["n"]) * dx
        w["Rs"] = R[cell % c["nR"]] + rng.uniform(-0.5, 0.5, c["n"]) * dR
    return w


def _params(c, w):
    return icwf.icwf_params(
        nx=w["nx"], nR=w["nR"], x_min=w["x_min"], x_max=w["x_max"], R_min=w["R_min"],
        R_max=w["R_max"], mass_x=w["mass_x"], mass_R=w["mass_R"], dt=w["dt"], n_traj=c.get("n", 1),
        precision=MODES[c.get("mode", "fp64")], svd_rel_cutoff=c.get("cutoff", 0.0),
        s_reg_eps=c.get("eps", 1e-6), coeff_scheme=int(c.get("frozen", False)), max_rank=0,
        solve_fp64=int(c.get("solve_fp64", False)), overlap_split=0)


def _job(c, seed):
    w = _problem(c, seed)
    sim = icwf.Icwf(_params(c, w), w["V"])
    sim.set_projectors(w["phi"])
    sim.init_from_positions(w["psi0"], w["xs"], w["Rs"])
    return sim


def _pool_jobs(c):
    """The jobs of a pool case as icwf cases, and what their names say: model, grid, ensemble."""
    out = []
    for name in c["jobs"].split(","):
        model, rest = ("cavity", name[3:]) if name.startswith("cav") else ("shin_metiu", name[2:])
        nx, nR, n = (int(v) for v in rest.split("x"))
        out.append(_icwf(name, model, nx, nR, n, "tf32x3", c["steps"]))
    return out


class _Pool:
    """A pool and its live jobs (which it owns); the program watches them between ticks."""

    def __init__(self, jobs):
        self.pool = icwf.icwf_pool_create(1 << 36, 8)
        self.jobs = []
        for sim in jobs:
            p = sim.p
            h = sim.release()
            icwf.icwf_pool_submit(self.pool, h, 1 << 40)
            self.jobs.append((h, p.nx, p.nR, p.n_traj))

    def __del__(self):
        icwf.icwf_pool_destroy(self.pool)


def prepare(case, seed):
    """An initialised handle (or pool of them): what a program holds before it starts stepping."""
    if case["kind"] == "pool":
        return case, _Pool([_job(c, 7 * seed + k) for k, c in enumerate(_pool_jobs(case))])
    if case["kind"] == "exact2d":
        w = _problem(case, seed)
        sim = icwf.Exact2D(_params(case, w), w["V"])
        sim.set_state(w["psi0"])
        sim.set_projectors(w["phi"])
        return case, sim
    return case, _job(case, seed)


# ---- a pass ------------------------------------------------------------------------------------

def _results(obs, st, mode):
    """Observables and trajectories (and CWFs, where read) in the precision the mode carries."""
    f, z = (np.float64, np.complex128) if mode == "fp64" else (np.float32, np.complex64)
    out = {"rho_x": obs["rho_x"].astype(f), "rho_R": obs["rho_R"].astype(f),
           "pop_decoh": np.concatenate([obs["pop"], obs["decoherence"].ravel()]).astype(f),
           "norm_energy": np.array([obs["norm"], obs["energy"]], dtype=f)}
    out.update({k: st[k].astype(f) for k in ("x", "R") if k in st})
    out.update({k: st[k].astype(z) for k in ("psi", "chi") if k in st})
    return out


def run(state):
    case, sim = state
    if case["kind"] == "pool":
        for _ in range(case["steps"]):
            icwf.icwf_pool_tick(sim.pool)
        return [_results(icwf.icwf_observables(h, nx, nR), icwf.icwf_get_state(h, n, nx, nR, cwfs=False), "tf32x3")
                for h, nx, nR, n in sim.jobs]
    sim.step(case["steps"])
    if case["kind"] == "exact2d":
        return _results(sim.observables(), {"psi": sim.state()}, "fp64")
    return _results(sim.observables(), sim.state(case["cwfs"]), case["mode"])


# ---- work --------------------------------------------------------------------------------------

def _rank(c):
    """Kept rank of the interaction (Shin-Metiu: about 15 at 1e-8 and 21 at 1e-12)."""
    if c["cutoff"] == 0.0:
        return min(c["nx"], c["nR"])
    return 1 if c["model"] == "cavity" else 15 if c["cutoff"] > 1e-10 else 21


def _fft_flops(nx, nR):
    return 5.0 * nx * nR * math.log2(nx * nR)


def work(case):
    """Bytes: the state (CWFs, positions, coefficients, S, Heff and the factor of S at t_n) read and
    written once per step, the observables' grid table V and projectors once.  Flops: the Hermitian
    Grams, factorisations, solves and products of the coefficient step, the propagations,
    velocities, and one reconstruction with its observables."""
    if case["kind"] == "pool":
        parts = [work(c) for c in _pool_jobs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nx, nR, s = case["nx"], case["nR"], case["steps"]
    n2 = nx * nR
    obs_flops = _fft_flops(nx, nR) + n2 * (12 + 4 * N_STATES)
    obs_bytes = 8.0 * n2 * (1 + N_STATES) + 8.0 * (nx + nR)
    if case["kind"] == "exact2d":
        return {"bytes": s * (2 * 16.0 + 8.0) * n2 + obs_bytes + 2 * 16.0 * n2,
                "flops": s * (2 * _fft_flops(nx, nR) + 18.0 * n2) + obs_flops}
    n, e = case["n"], 16.0 if case["mode"] == "fp64" else 8.0
    gram = 4.0 * n * n * (_rank(case) + 1) * (nx + nR)
    chol = (1 if case["frozen"] else 2) * 4.0 / 3.0 * n ** 3
    coeff = 4 * (8.0 * n * n + 2 * 4.0 * n * n)
    fft = 2 * 5.0 * n * (nx * math.log2(nx) + nR * math.log2(nR)) + 20.0 * n * (nx + nR)
    vel = n * n * 90.0
    step_bytes = 2 * (e * n * (nx + nR) + 32.0 * n + 3 * 16.0 * n * n)
    return {"bytes": s * step_bytes + e * n * (nx + nR) + obs_bytes,
            "flops": s * (gram + chol + coeff + fft + vel) + 8.0 * n * n2 + obs_flops}


# ---- 64-bit values -----------------------------------------------------------------------------

def _exact_obs(Psi, w, dev):
    T = lambda a: torch.as_tensor(a, device=dev)  # noqa: E731
    dx, dR, nx, nR = w["dx"], w["dR"], w["nx"], w["nR"]
    dens = Psi.real ** 2 + Psi.imag ** 2
    kx = T(2 * np.pi * np.fft.fftfreq(nx, dx))
    kR = T(2 * np.pi * np.fft.fftfreq(nR, dR))
    ek = dR * dx / nx * ((torch.fft.fft(Psi, dim=0).abs() ** 2) * (kx * kx / (2 * w["mass_x"]))[:, None]).sum()
    ek = ek + dx * dR / nR * ((torch.fft.fft(Psi, dim=1).abs() ** 2) * (kR * kR / (2 * w["mass_R"]))[None, :]).sum()
    norm = dx * dR * dens.sum()
    energy = (ek + dx * dR * (dens * T(w["V"])).sum()) / norm
    ch = dx * torch.einsum("nji,ij->nj", T(w["phi"]).to(Psi.dtype), Psi)
    pn = ch.abs() ** 2
    h = lambda t: t.cpu().numpy()  # noqa: E731
    return {"rho_x": h(dR * dens.sum(1)), "rho_R": h(dx * dens.sum(0)), "pop": h(dR * pn.sum(1)),
            "decoherence": h(dR * pn @ pn.T), "norm": float(norm), "energy": float(energy)}


def _stencil(p, lo, d, n):
    """4-point cubic Lagrange stencils at the positions p: start index, weights, derivative weights."""
    s = (p - lo) / d - 0.5
    i0 = torch.clamp(torch.floor(s).long() - 1, 0, n - 4)
    u = s - i0
    a, b, c = u - 1, u - 2, u - 3
    w = torch.stack([-a * b * c / 6, u * b * c / 2, -u * a * c / 2, u * a * b / 6])
    dw = torch.stack([-(b * c + a * c + a * b) / 6, (b * c + u * c + u * b) / 2,
                      -(a * c + u * c + u * a) / 2, (a * b + u * b + u * a) / 6]) / d
    return i0, w, dw


def _at(f, st, deriv=False):
    """f[:, ...] (grid first) at the stencils: (points, ...)."""
    i0, w, dw = st
    c = dw if deriv else w
    return sum(f[i0 + m] * c[m].reshape([-1] + [1] * (f.dim() - 1)) for m in range(4))


def _exact_icwf(c, w, dev):
    """The ICWF steps of one job in complex128: cubic Lagrange slices and velocities, Strang steps at
    the midpoints, the rank-k matrix elements, RK4 with S + eps I solves."""
    T = lambda a: torch.as_tensor(a, device=dev)  # noqa: E731
    dx, dR, nx, nR, dt, n = w["dx"], w["dR"], w["nx"], w["nR"], w["dt"], c["n"]
    V, psi0 = T(w["V"]), T(w["psi0"])
    v1 = V.mean(1)
    v2 = V.mean(0) - V.mean()
    U, s, Wt = torch.linalg.svd((V - v1[:, None] - v2[None, :]).cpu(), full_matrices=False)
    tails = torch.sqrt(torch.flip(torch.cumsum(torch.flip(s * s, [0]), 0), [0]))
    k = len(s) if c["cutoff"] <= 0 else max(1, int((tails > c["cutoff"] * tails[0]).sum()))
    u, wk, s = U[:, :k].to(dev), Wt[:k].T.to(dev), s[:k].to(dev)
    sx = lambda p: _stencil(p, w["x_min"], dx, nx)  # noqa: E731
    sR = lambda p: _stencil(p, w["R_min"], dR, nR)  # noqa: E731
    x, R = T(w["xs"]), T(w["Rs"])
    psi = _at(psi0.T, sR(R)).T.contiguous()          # nx x n
    chi = _at(psi0, sx(x)).T.contiguous()            # nR x n
    psi = psi / torch.sqrt(dx * (psi.abs() ** 2).sum(0))
    chi = chi / torch.sqrt(dR * (chi.abs() ** 2).sum(0))
    eye = torch.eye(n, dtype=psi.dtype, device=dev)

    def matrices(psi, chi, x, R):
        S1, S2 = dx * psi.mH @ psi, dR * chi.mH @ chi
        S = S1 * S2
        tx, tR = sx(x), sR(R)
        ux, wR = _at(u, tx), _at(wk, tR)
        d = _at(v1, tx) + _at(v2, tR) + (ux * wR) @ s
        H = -S * d[None, :]
        for q in range(k):
            A = dx * psi.mH @ (u[:, q, None] * psi) - S1 * ux[None, :, q]
            B = dR * chi.mH @ (wk[:, q, None] * chi) - S2 * wR[None, :, q]
            H += s[q] * A * B
        return S, H

    def solver(S):
        L = torch.linalg.cholesky(S + c["eps"] * eye)
        return lambda y: torch.cholesky_solve(y[:, None], L)[:, 0]

    def strang(f, v, d, mass):
        kk = T(2 * np.pi * np.fft.fftfreq(f.shape[0], d))
        half = torch.exp(-0.5j * dt * v)
        return half * torch.fft.ifft(torch.exp(-0.5j * dt * kk * kk / mass)[:, None] * torch.fft.fft(half * f, dim=0), dim=0)

    S, H = matrices(psi, chi, x, R)
    inv = solver(S)
    C = inv(dx * dR * (psi.conj() * (psi0 @ chi.conj())).sum(0))
    for _ in range(c["steps"]):
        tx, tR = sx(x), sR(R)
        E1, G1, E2, G2 = _at(psi, tx), _at(psi, tx, True), _at(chi, tR), _at(chi, tR, True)
        den = (E1 * E2) @ C
        xn = x + dt * (((G1 * E2) @ C) / den).imag / w["mass_x"]
        Rn = R + dt * (((E1 * G2) @ C) / den).imag / w["mass_R"]
        xn = torch.clamp(xn, float(w["x"][0]), float(w["x"][-1]))
        Rn = torch.clamp(Rn, float(w["R"][0]), float(w["R"][-1]))
        Ve = _at(V.T.contiguous(), sR(0.5 * (R + Rn))).T
        Vn = _at(V, sx(0.5 * (x + xn))).T
        psi, chi = strang(psi, Ve, dx, w["mass_x"]), strang(chi, Vn, dR, w["mass_R"])
        x, R = xn, Rn
        Sn, Hn = matrices(psi, chi, x, R)
        invn = solver(Sn)
        if c["frozen"]:
            stages = [(inv, H)] * 4
        else:
            mid = (solver(0.5 * (S + Sn)), 0.5 * (H + Hn))
            stages = [(inv, H), mid, mid, (invn, Hn)]
        ks = []
        for (f, M), h in zip(stages, (0.0, 0.5 * dt, 0.5 * dt, dt)):
            ks.append(-1j * f(M @ (C + h * ks[-1] if ks else C)))
        C = C + dt / 6 * (ks[0] + 2 * ks[1] + 2 * ks[2] + ks[3])
        S, H, inv = Sn, Hn, invn
    obs = _exact_obs((psi * C) @ chi.T, w, dev)
    st = {"x": x.cpu().numpy(), "R": R.cpu().numpy()}
    if c["cwfs"]:
        st.update(psi=psi.cpu().numpy(), chi=chi.cpu().numpy())
    return obs, st


def exact(case, seed):
    dev = _device()
    if case["kind"] == "pool":
        return [_results(*_exact_icwf(c, _problem(c, 7 * seed + k), dev), "fp64")
                for k, c in enumerate(_pool_jobs(case))]
    w = _problem(case, seed)
    if case["kind"] == "icwf":
        return _results(*_exact_icwf(case, w, dev), "fp64")
    T = lambda a: torch.as_tensor(a, device=dev)  # noqa: E731
    kx = T(2 * np.pi * np.fft.fftfreq(w["nx"], w["dx"]))
    kR = T(2 * np.pi * np.fft.fftfreq(w["nR"], w["dR"]))
    half = torch.exp(-0.5j * case["dt"] * T(w["V"]))
    kin = torch.exp(-0.5j * case["dt"] * (kx[:, None] ** 2 / w["mass_x"] + kR[None, :] ** 2 / w["mass_R"]))
    Psi = T(w["psi0"])
    for _ in range(case["steps"]):
        Psi = half * torch.fft.ifft2(kin * torch.fft.fft2(half * Psi))
    return _results(_exact_obs(Psi, w, dev), {"psi": Psi.cpu().numpy()}, "fp64")
