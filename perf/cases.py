"""Timed cases of the lattice Dyson solver, through the Python binding that programs use.

A case is a dict of plain values with a "kind":

  solve      block columns of one lattice: build Lambda (build = True), solve, read the
             observables; with g = True the block columns G are written to the caller's buffer
  batch      uneven instances, one block column each, as one Batch
  adjoint    loss and gradients of sum_i w_i n_i(t) (+ v_i D_i(t)) from the transposed solve
  selfenergy iterations of the self-consistency loop: local Green's functions of every site,
             self-energy step

Sizes and drives are those of workloads/, of the tests and of the benchmark, or lie between them.
`precision` 0 is the FP64 series, 1 the mixed-precision solve; `variant` is the sweep form a
program has selected (0: the default, 2: the fused form that the autotuner picks).
"""
import math
import random

import numpy as np
import torch

import workloads as wl
from paper_1309_5994_gb300 import binding

DEV = "cuda:0"


def listed():
    return [
        # the smallest calls: a parameter scan over tiny clusters, every source, an odd contour;
        # latency and launches count
        dict(name="f64_3x3_nc26", kind="solve", Lx=3, Ly=3, Nt=10, Nm=6, beta=1.0, U=10.0, trap=0.3, drive=True,
             disorder=False, precision=0, tol=1e-12, columns=9, build=True, g=True, variant=0),
        # the 4x4 benchmark configuration: all sixteen sources in FP64
        dict(name="f64_4x4_nc64", kind="solve", Lx=4, Ly=4, Nt=24, Nm=16, beta=1.0, U=20.0, trap=0.5, drive=False,
             disorder=False, precision=0, tol=1e-12, columns=16, build=True, g=True, variant=0),
        # the plain FP64 series at a size where arithmetic counts: the validation arm of a
        # mixed-precision run, and the precision of the self-consistency loop
        dict(name="f64_10x10_nc128", kind="solve", Lx=10, Ly=10, Nt=48, Nm=32, beta=2.0, U=20.0, trap=0.05,
             drive=True, disorder=False, precision=0, tol=1e-12, columns=4, build=False, g=True, variant=0),
        # an ordinary mixed-precision call by a program that selects nothing: default sweep form,
        # tight tolerance
        dict(name="mixed_8x8_nc128", kind="solve", Lx=8, Ly=8, Nt=48, Nm=32, beta=2.0, U=20.0, trap=0.05, drive=True,
             disorder=False, precision=1, tol=1e-10, columns=8, build=False, g=True, variant=0),
        # a rectangular lattice on a contour that is no multiple of any tile
        dict(name="mixed_9x7_nc100", kind="solve", Lx=9, Ly=7, Nt=38, Nm=24, beta=2.0, U=18.0, trap=0.05, drive=True,
             disorder=False, precision=1, tol=1e-10, columns=6, build=False, g=True, variant=0),
        # every site and bond with its own noisy values (disorder), tight tolerance, G to the caller;
        # the series converges slowly there and hands over to GMRES
        dict(name="mixed_disorder_10x10_nc256", kind="solve", Lx=10, Ly=10, Nt=112, Nm=32, beta=2.0, U=20.0,
             trap=0.02, drive=False, disorder=True, precision=1, tol=1e-10, columns=4, build=False, g=True, variant=2),
        # the benchmark's step: build Lambda, sixteen block columns, observables
        dict(name="mixed_16x16_nc256", kind="solve", Lx=16, Ly=16, Nt=112, Nm=32, beta=2.0, U=20.0, trap=0.02,
             drive=False, disorder=False, precision=1, tol=1e-6, columns=16, build=True, g=False, variant=2),
        # a driven lattice on the long contour, where the FP32 series gives way to GMRES
        dict(name="mixed_driven_12x12_nc384", kind="solve", Lx=12, Ly=12, Nt=160, Nm=64, beta=2.0, U=20.0,
             trap=0.005, drive=True, disorder=False, precision=1, tol=1e-6, columns=1, build=False, g=True,
             variant=2),
        # a scan over uneven traps and drives in one batch
        dict(name="batch_uneven_6", kind="batch", count=6, Lmin=8, Lmax=16, tol=1e-10),
        # gradient of a small lattice's densities and double occupancies, as an optimiser's inner step
        dict(name="adjoint_obs_5x4_nc48", kind="adjoint", Lx=5, Ly=4, Nt=18, Nm=12, beta=1.0, U=12.0, trap=0.2,
             docc=True, precision=0, tol=1e-12, variant=0),
        # the 24x24 gradient configuration
        dict(name="adjoint_24x24_nc256", kind="adjoint", Lx=24, Ly=24, Nt=96, Nm=64, beta=2.0, U=20.0, trap=0.005,
             docc=False, precision=1, tol=1e-10, variant=2),
        # two iterations of the self-consistency loop of the driven 8x8 lattice
        dict(name="selfenergy_8x8_nc64", kind="selfenergy", Lx=8, Ly=8, Nt=24, Nm=16, beta=2.0, U=20.0, trap=0.05,
             iterations=2, tol=1e-10),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _contour(rng, lo, hi, multiple):
    """(Nt, Nm) with Nc = 2 Nt + Nm in lo..hi, Nm about Nc/8..Nc/3; Nc a multiple of `multiple`."""
    nc = max(multiple, _log_int(rng, lo, hi) // multiple * multiple)
    nm = max(2, int(nc * rng.uniform(0.125, 0.33)))
    nm -= (nc - nm) % 2
    return (nc - nm) // 2, max(nm, 1 if nc % 2 else 2)


def draw(rng):
    kind = rng.choice(["f64", "f64", "mixed", "mixed", "mixed", "ragged", "batch", "adjoint", "selfenergy"])
    U, trap = round(rng.uniform(16.0, 28.0), 3), round(rng.uniform(0.005, 0.3), 4)
    drive, disorder = rng.random() < 0.6, rng.random() < 0.3
    Lx = _log_int(rng, 2, 16)
    Ly = min(16, max(1, Lx + rng.choice([-1, 0, 0, 1, 2])))
    beta = rng.choice([1.0, 2.0])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 8), Lmin=rng.randint(3, 8), Lmax=rng.randint(9, 16),
                    tol=rng.choice([1e-6, 1e-10]))
    if kind == "adjoint":
        if rng.random() < 0.5:
            Nt, Nm = _contour(rng, 16, 96, 1)
            L = _log_int(rng, 2, 6)
            return dict(kind="adjoint", Lx=L, Ly=max(1, L - rng.randint(0, 1)), Nt=Nt, Nm=Nm, beta=beta, U=U,
                        trap=trap, docc=rng.random() < 0.5, precision=rng.choice([0, 1]), tol=1e-11, variant=0)
        Nt, Nm = _contour(rng, 128, 256, 64)
        return dict(kind="adjoint", Lx=min(Lx, 16), Ly=Ly, Nt=Nt, Nm=Nm, beta=2.0, U=U, trap=trap,
                    docc=rng.random() < 0.3, precision=1, tol=1e-10, variant=2)
    if kind == "selfenergy":
        Nt, Nm = _contour(rng, 16, 64, 1)
        L = _log_int(rng, 2, 8)
        return dict(kind="selfenergy", Lx=L, Ly=max(1, L - rng.randint(0, 1)), Nt=Nt, Nm=Nm, beta=beta, U=U,
                    trap=trap, iterations=2, tol=1e-10)
    if kind == "f64":
        Nt, Nm = _contour(rng, 16, 192, rng.choice([1, 1, 64]))
        precision, tol, most = 0, 1e-12, 1.2e10
    elif kind == "ragged":
        Nt, Nm = _contour(rng, 32, 250, 1)
        precision, tol, most = 1, rng.choice([1e-6, 1e-10]), 4e10
    else:
        Nt, Nm = _contour(rng, 64, 256, 64)
        precision, tol, most = 1, rng.choice([1e-6, 1e-10]), 4e11
    nc = 2 * Nt + Nm
    columns = _log_int(rng, 1, 16)
    per = 8.0 * nc ** 3 * Lx * Ly
    columns = max(1, min(columns, Lx * Ly, int(most / per)))
    while columns == 1 and 8.0 * nc ** 3 * Lx * Ly > most and Lx > 2:
        Lx, Ly = Lx - 1, max(1, Ly - 1)
    g = columns * Lx * Ly * nc * nc * 16 <= 1 << 30
    return dict(kind="solve", Lx=Lx, Ly=Ly, Nt=Nt, Nm=Nm, beta=beta, U=U, trap=trap, drive=drive, disorder=disorder,
                precision=precision, tol=tol, columns=columns, build=rng.random() < 0.5, g=g,
                variant=rng.choice([0, 2]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _problem(case, seed):
    """The lattice of a case: the seed moves U, the trap, the chemical potential, the drive's phase."""
    r = np.random.default_rng(seed)
    drive = case.get("drive", True)
    p = wl.uniform_problem(
        "case", case["Lx"], case["Nt"], case["Nm"], 0.05, case["beta"], float(r.uniform(-0.5, 0.5)),
        case["trap"] * float(r.uniform(0.9, 1.1)), case["U"] * float(r.uniform(0.97, 1.03)), 1.0, Ly=case["Ly"],
        aU=0.1 if drive else 0.0, aJ=0.2 if drive else 0.0, omega=20.0 if drive else 0.0,
        phase=float(r.uniform(0.0, 2.0 * np.pi)))
    return wl.random_tables(p, seed + 1, 0.05) if case.get("disorder") else p


def _instances(case, seed):
    """Uneven instances: sides and contours from the case, the physics from the seed."""
    shape = random.Random("%d %d %d" % (case["count"], case["Lmin"], case["Lmax"]))
    r = np.random.default_rng(seed)
    out = []
    for k in range(case["count"]):
        L = shape.randint(case["Lmin"], case["Lmax"])
        nc = shape.choice([128, 192, 256])
        out.append(wl.uniform_problem("case%d" % k, L, (nc - nc // 4) // 2, nc // 4, 0.05, 2.0, 0.0,
                                      float(r.uniform(0.005, 0.05)), float(r.uniform(16.0, 30.0)), 1.0,
                                      aU=0.1, aJ=0.2, omega=20.0, phase=float(r.uniform(0.0, 2.0 * np.pi))))
    return out


def _sources(case, p):
    """Source sites of a solve: spread over the lattice by a fixed rule."""
    return [int(s) for s in wl.sample_sources(p.Nr, case["columns"], 7)]


def _solver(p, variant):
    s = binding.Solver(p, device=0)
    if variant:
        s.set_sweep_variant(variant)
    return s


def _c128(*shape):
    return torch.zeros(shape, dtype=torch.complex128, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ps = _instances(case, seed)
        solvers = [_solver(p, 0) for p in ps]
        for s in solvers:
            s.build_sigma()
        return dict(case=case, solvers=solvers, batch=binding.Batch(solvers), sources=[[p.Nr // 2] for p in ps],
                    g=[_c128(1, p.Nr, p.Nc, p.Nc) for p in ps])
    p = _problem(case, seed)
    st = dict(case=case, solver=_solver(p, case.get("variant", 0)))
    if kind == "solve":
        st["sources"] = _sources(case, p)
        st["g"] = _c128(len(st["sources"]), p.Nr, p.Nc, p.Nc) if case["g"] else None
        if not case["build"]:
            st["solver"].build_sigma()
    elif kind == "adjoint":
        r = np.random.default_rng(seed + 2)
        st["w"] = r.uniform(0.0, 1.0, p.Nr)
        st["v"] = r.uniform(0.0, 1.0, p.Nr) if case["docc"] else None
        st["solver"].build_sigma()
    else:
        st["gloc"] = [_c128(p.Nr, p.Nc, p.Nc) for _ in range(case["iterations"])]
        st["sigma"] = [_c128(p.Nr, p.Nc, p.Nc) for _ in range(case["iterations"])]
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind, tol = case["kind"], case["tol"]
    if kind == "batch":
        st["batch"].solve(st["sources"], tol=tol, g_outs=st["g"])
        return st["g"]
    s = st["solver"]
    if kind == "solve":
        if case["build"]:
            s.build_sigma()
        s.solve(st["sources"], precision=case["precision"], tol=tol, g_out=st["g"])
        n, ekin, docc = s.observables()
        rows = st["sources"]
        out = dict(n=n[rows], ekin=ekin[rows], docc=docc[rows])
        if st["g"] is not None:
            out["g"] = st["g"]
        return out
    if kind == "adjoint":
        if st["v"] is None:
            loss, gU, gJ, _ = s.adjoint(st["w"], precision=case["precision"], tol=tol)
        else:
            loss, gU, gJ, _ = s.adjoint_obs(st["w"], st["v"], precision=case["precision"], tol=tol)
        return dict(loss=loss, gU=gU, gJ=gJ)
    s.build_sigma()
    out = {}
    for k in range(case["iterations"]):
        s.local_greens(precision=binding.PREC_F64, tol=tol, out=st["gloc"][k])
        out["measure%d" % k] = s.selfenergy_step(st["gloc"][k], sigma_tilde=st["sigma"][k])
        out["gloc%d" % k], out["sigma%d" % k] = st["gloc"][k], st["sigma"][k]
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _terms(Nt, tol):
    """Terms of the series to `tol`: the hopping series of a real branch of length T decays like (2 sqrt(2) T)^n / n!."""
    x, n, log = 2.0 * math.sqrt(2.0) * 0.05 * Nt, 0, 0.0
    while n < 4 or log > math.log(tol):
        n += 1
        log += math.log(max(x, 1.0) / n)
    return n


def _sweeps(Nr, Nt, Nm, columns, tol):
    """Flops of `columns` vector columns: one complex Nc x Nc product per site, column and term."""
    nc = 2 * Nt + Nm
    return 8.0 * nc * nc * Nr * columns * _terms(Nt, tol)


def work(case):
    kind, tol = case["kind"], case["tol"]
    if kind == "batch":
        ps = _instances(case, 0)
        return dict(flops=sum(_sweeps(p.Nr, p.Nt, p.Nm, p.Nc, tol) for p in ps),
                    bytes=sum(32.0 * p.Nr * p.Nc ** 2 for p in ps))       # Lambda read, G written
    Nr, Nt, Nm = case["Lx"] * case["Ly"], case["Nt"], case["Nm"]
    nc, nb = 2 * Nt + Nm, wl.n_bonds(case["Lx"], case["Ly"])
    tables = 8.0 * (Nr + nb) * Nt
    lam = 16.0 * Nr * nc * nc
    if kind == "solve":
        out = lam * case["columns"] if case["g"] else 0.0
        return dict(flops=_sweeps(Nr, Nt, Nm, case["columns"] * nc, tol),
                    bytes=lam + out + tables + 24.0 * case["columns"] * Nt)
    if kind == "adjoint":
        return dict(flops=_sweeps(Nr, Nt, Nm, (3 if case["docc"] else 2) * Nr, tol), bytes=lam + 2 * tables)
    it = case["iterations"]
    # per iteration: Nr block columns, the cumulant contraction (16 Nm + 64) Nc^3 per site, and
    # the local solve (LU and two products of complex Nc x Nc blocks)
    return dict(flops=it * (_sweeps(Nr, Nt, Nm, Nr * nc, tol) + Nr * nc ** 3 * (16.0 * Nm + 64 + 8 * (2 / 3 + 2))),
                bytes=it * 4 * lam + tables)


def tolerance(case):
    """An iterative solve that stops at another sweep differs by about the tolerance that the call asks
    for, docc by a few times that (its difference quotient).  Measured against exact(): up to 0.2 of
    it in FP64 and at 1e-10, 3 times it at 1e-6; four times the latter is stated for all.  The
    second self-consistency iteration carries the first one's differences through two local inverses."""
    return dict(rel=(100 if case["kind"] == "selfenergy" else 12) * case["tol"])


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _tables64(p, U, J):
    """eps [Nr], Lambda [Nr, Nc, Nc], weights [Nc], real-time index of each contour point."""
    Nt, Nm, nc = p.Nt, p.Nm, p.Nc
    f64 = dict(dtype=torch.float64, device=U.device)
    y, x = torch.meshgrid(torch.arange(p.Ly, **f64), torch.arange(p.Lx, **f64), indexing="ij")
    r2 = ((x - 0.5 * (p.Lx - 1)) ** 2 + (y - 0.5 * (p.Ly - 1)) ** 2).reshape(-1)
    eps = p.trap_c * r2 - 0.5 * U[:, 0] - p.mu
    logw = -p.beta * torch.stack([torch.zeros_like(eps), eps, eps, 2 * eps + U[:, 0]], 1)
    logw = logw - torch.logsumexp(logw, 1, keepdim=True)
    k = torch.arange(Nt, device=U.device)
    time = torch.cat([k, k.flip(0), torch.zeros(Nm, dtype=torch.long, device=U.device)])
    w = torch.cat([torch.full((Nt,), p.dt, **f64), torch.full((Nt,), -p.dt, **f64), torch.zeros(Nm, **f64)]) + 0j
    w[2 * Nt:] = -1j * p.beta / Nm
    idx = torch.arange(nc, device=U.device)
    later = idx[:, None] > idx[None, :]
    back = idx[Nt:2 * Nt]
    later[back, back] = True
    tau = torch.arange(Nm, **f64) * (p.beta / Nm)
    lam = 0
    for E, la, lb in ((eps[:, None].expand(-1, Nt), logw[:, 0], logw[:, 1]), (eps[:, None] + U, logw[:, 1], logw[:, 3])):
        phi = torch.cumsum(E, 1) * p.dt - E * p.dt
        phi = torch.cat([phi, phi.flip(1), torch.zeros(len(eps), Nm, **f64)], 1) + 0j
        phi = torch.cat([phi[:, :2 * Nt], -1j * tau[None, :] * E[:, :1]], 1)
        d = -1j * (phi[:, :, None] - phi[:, None, :])
        lam = lam + torch.where(later, torch.exp(la[:, None, None] + d), -torch.exp(lb[:, None, None] + d))
    return eps, -1j * lam, w, time


def _bonds(p):
    h = [(y * p.Lx + x, y * p.Lx + x + 1) for y in range(p.Ly) for x in range(p.Lx - 1)]
    v = [(y * p.Lx + x, (y + 1) * p.Lx + x) for y in range(p.Ly - 1) for x in range(p.Lx)]
    return h + v


def _device64(p):
    dev = DEV if torch.cuda.is_available() else "cpu"
    return (torch.tensor(p.U, device=dev), torch.tensor(p.J.reshape(-1, p.Nt), device=dev))


def _series64(p, lam, JW, cols):
    """G [Nr, Nc, n] of the vector columns (site, time): the series, all sites at once."""
    n = len(cols)
    B = torch.zeros((p.Nr, p.Nc, n), dtype=torch.complex128, device=lam.device)
    sites = torch.tensor([c[0] for c in cols], device=lam.device)
    times = torch.tensor([c[1] for c in cols], device=lam.device)
    B[sites, :, torch.arange(n, device=lam.device)] = lam[sites, :, times]
    bonds = _bonds(p)
    G, top, best, flat = B.clone(), float(B.abs().max()), math.inf, 0
    for _ in range(400):
        X = torch.zeros_like(G)
        for b, (i, j) in enumerate(bonds):
            X[i].addcmul_(JW[b][:, None], G[j])
            X[j].addcmul_(JW[b][:, None], G[i])
        new = B + torch.bmm(lam, X)
        upd = float((new - G).abs().max()) / top
        G = new
        flat = 0 if upd < 0.7 * best else flat + 1
        best = min(best, upd)
        if upd < 1e-14 or (best < 1e-8 and flat > 3):
            break
    return G


def _columns64(p, sources, need_g):
    """Per source (site): G columns as [Nr, Nc, Nc] (all times) or [Nr, Nc, Nt] (forward times only)."""
    U, J = _device64(p)
    eps, lam, w, time = _tables64(p, U, J)
    JW = J[:, time] * w[None, :]
    m = p.Nc if need_g else p.Nt
    G = _series64(p, lam, JW, [(s, z) for s in sources for z in range(m)])
    n, ekin, docc = (np.full((len(sources), p.Nt), np.nan) for _ in range(3))
    k = torch.arange(p.Nt, device=G.device)
    bonds = _bonds(p)
    for q, s in enumerate(sources):
        C = G[:, :, q * m:(q + 1) * m]
        geq = C[s][k, k]
        acc = torch.zeros_like(geq)
        for b, ij in enumerate(bonds):
            if s in ij:
                acc = acc + J[b] * C[ij[0] + ij[1] - s][k, k]
        dens, kin = geq.imag, acc.imag
        dre = (geq[1:] - C[s][k[:-1], k[1:]]).real / p.dt
        n[q], ekin[q] = dens.cpu().numpy(), kin.cpu().numpy()
        docc[q, 1:] = ((dre - eps[s] * dens[1:] - kin[1:]) / U[s, 1:]).cpu().numpy()
    g = G.reshape(p.Nr, p.Nc, len(sources), m).permute(2, 0, 1, 3).contiguous() if need_g else None
    return dict(n=n, ekin=ekin, docc=docc), g


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_columns64(p, [p.Nr // 2], True)[1] for p in _instances(case, seed)]
    p = _problem(case, seed)
    if kind == "solve":
        obs, g = _columns64(p, _sources(case, p), case["g"])
        if g is not None:
            obs["g"] = g
        return obs
    if kind == "selfenergy":
        # the first iteration's local Green's functions; the steps after it have no short plain form
        U, J = _device64(p)
        _, lam, w, time = _tables64(p, U, J)
        G = _series64(p, lam, J[:, time] * w[None, :], [(s, z) for s in range(p.Nr) for z in range(p.Nc)])
        out = {"%s%d" % (n, k): None for n in ("measure", "gloc", "sigma") for k in range(case["iterations"])}
        out["gloc0"] = torch.stack([G[s][:, s * p.Nc:(s + 1) * p.Nc] for s in range(p.Nr)])
        return out
    if p.Nr * p.Nc > 2048:
        return None                                        # the dense gradient below would take too long
    # the gradient by torch's reverse mode through the dense solve
    r = np.random.default_rng(seed + 2)
    wn = r.uniform(0.0, 1.0, p.Nr)
    wd = r.uniform(0.0, 1.0, p.Nr) if case["docc"] else np.zeros(p.Nr)
    U, J = (t.requires_grad_(True) for t in _device64(p))
    eps, lam, w, time = _tables64(p, U, J)
    JW = J[:, time] * w[None, :]
    nc, kf = p.Nc, p.Nt - 1
    A = torch.eye(p.Nr * nc, dtype=torch.complex128, device=U.device).reshape(p.Nr, nc, p.Nr, nc).clone()
    for b, (i, j) in enumerate(_bonds(p)):
        A[i, :, j, :] = -lam[i] * JW[b][None, :]
        A[j, :, i, :] = -lam[j] * JW[b][None, :]
    B = torch.zeros((p.Nr, nc, p.Nr), dtype=torch.complex128, device=U.device)
    for i in range(p.Nr):
        B[i, :, i] = lam[i][:, kf]
    G = torch.linalg.solve(A.reshape(p.Nr * nc, -1), B.reshape(p.Nr * nc, -1)).reshape(p.Nr, nc, p.Nr)
    loss = 0.0
    for i in range(p.Nr):
        geq = G[i, kf, i]
        dens = geq.imag
        kin = sum((J[b, kf] * G[a + c - i, kf, i] for b, (a, c) in enumerate(_bonds(p)) if i in (a, c)),
                  torch.zeros_like(geq)).imag
        d = ((geq - G[i, kf - 1, i]).real / p.dt - eps[i] * dens - kin) / U[i, kf]
        loss = loss + wn[i] * dens + wd[i] * d
    gU, gJ = torch.autograd.grad(loss, (U, J), allow_unused=True)
    gJ = torch.zeros_like(J) if gJ is None else gJ
    return dict(loss=float(loss.detach()), gU=gU.cpu().numpy(), gJ=gJ.cpu().numpy())
