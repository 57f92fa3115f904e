"""The calls whose speed this repository is held to, with what they read, do and should return.

Each case is one public call (or the few that belong together) of ``paper_1706_02145_gb300`` as a program that
uses it makes them, on seeded sphere packings with the sizes, radii, indices and wavelengths of the repository's
own workloads: clusters of tens of spheres, the 10 000-sphere polydisperse slab at lmax 4, the 100 000-sphere slab
at lmax 3 and ensembles of 200 to 3000 spheres with lmax 2 to 5.

``exact`` restates what the calls return in plain torch in 64 bits (the printed addition-theorem coefficients,
Mie series, angular-spectrum integrals and field expansions), without the package.
"""

import math
from fractions import Fraction
from functools import lru_cache

import numpy as np
import torch

import paper_1706_02145_gb300 as celes
from paper_1706_02145_gb300 import binding

RADIUS_SIGMA = 0.1  # ln R of the polydisperse packings


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one product on a 50-sphere cluster, where the launches count
        dict(name="coupling_50", kind="matvec", op="coupling", precision="fp32", N=50, lmax=3, nrhs=1, poly=False,
             wavelength=550.0, index_re=1.52, index_im=0.0),
        # one ensemble's operator at the highest degree with its eight plane waves, odd size
        dict(name="master_777_l5_rhs8", kind="matvec", op="master", precision="fp32", N=777, lmax=5, nrhs=8,
             poly=False, wavelength=633.0, index_re=1.8, index_im=0.0),
        # the Krylov operator of the polydisperse slab, the bulk of every solve
        dict(name="master_slab_10000", kind="matvec", op="master", precision="fp32", N=10000, lmax=4, nrhs=1,
             poly=True, wavelength=550.0, index_re=1.5, index_im=0.001),
        # the largest workload: the 100 000-sphere monodisperse slab
        dict(name="coupling_large_100000", kind="matvec", op="coupling", precision="fp32", N=100000, lmax=3, nrhs=1,
             poly=False, wavelength=550.0, index_re=1.52, index_im=0.0),
        # the FP64 residual of the refinement
        dict(name="master_fp64_2001", kind="matvec", op="master", precision="fp64", N=2001, lmax=4, nrhs=1, poly=True,
             wavelength=550.0, index_re=1.5, index_im=0.001),
        # the operator of a lockstep batch: ensembles of mixed degree and size, several plane waves each
        dict(name="batch_12x4", kind="batch", precision="fp32", ensembles=12, rhs=4, n_lo=200, n_hi=1200),
        # preconditioner: factorisation of the diagonal blocks, then its application in FP64
        dict(name="precond_build_1500", kind="precond_build", precision="fp64", N=1500, lmax=4, nrhs=1, poly=True,
             edge=1000.0, wavelength=550.0, index_re=1.5, index_im=0.001),
        # one application per Krylov step
        dict(name="precond_apply_5000", kind="precond_apply", precision="fp32", N=5000, lmax=3, nrhs=1, poly=False,
             edge=870.0, wavelength=550.0, index_re=1.52, index_im=0.0),
        # from host arrays to T-matrices and Gaussian-beam coefficients back on the host
        dict(name="setup_gaussian_10000", kind="setup", beam="gaussian", N=10000, lmax=4, nrhs=1, poly=True,
             wavelength=550.0, index_re=1.5, index_im=0.001),
        # scattered amplitudes of the slab on a hemisphere grid
        dict(name="farfield_10000x2048", kind="farfield", N=10000, lmax=4, directions=2048, poly=True,
             wavelength=550.0, index_re=1.5, index_im=0.001),
        # total field on a plane through a cluster in a Gaussian beam
        dict(name="nearfield_1000x4096", kind="nearfield", beam="gaussian", N=1000, lmax=3, points=4096, poly=False,
             wavelength=550.0, index_re=1.52, index_im=0.0),
        # a whole solve of a small cluster, refined until its answer does not depend on the path to it
        dict(name="solve_120", kind="solve", mode="mixed", solver="gmres", N=120, lmax=3, nrhs=1, edge=0.0, poly=False,
             wavelength=550.0, index_re=1.52, index_im=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds, over their whole ranges."""
    kind = rng.choice(["matvec", "matvec", "matvec", "matvec", "batch", "precond_build", "precond_apply", "setup",
                       "farfield", "nearfield", "solve"])
    poly = rng.random() < 0.5
    # cuboids of up to about three spheres along an edge
    edge = round(rng.uniform(500.0, 1200.0) if poly else rng.uniform(250.0, 550.0), 1)
    optics = dict(poly=poly, wavelength=round(rng.uniform(400.0, 800.0), 1), index_re=round(rng.uniform(1.45, 2.0), 3),
                  index_im=rng.choice([0.0, 0.001]))
    if kind == "matvec":
        precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        lmax = rng.randint(1, 5)
        N = _log_int(rng, 20, 30000 if precision == "fp32" else 3000)
        nrhs = rng.choice([1, 1, 2, 8]) if N < 3000 else 1
        return dict(kind=kind, op=rng.choice(["coupling", "master"]), precision=precision, N=N, lmax=lmax, nrhs=nrhs,
                    **optics)
    if kind == "batch":
        hi = rng.randint(300, 1500)
        return dict(kind=kind, precision=rng.choice(["fp32", "fp32", "fp64"]) if hi < 500 else "fp32",
                    ensembles=rng.randint(2, 16), rhs=rng.randint(1, 8), n_lo=rng.randint(20, 200), n_hi=hi)
    if kind == "precond_build":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp64"]), N=_log_int(rng, 50, 1500),
                    lmax=rng.randint(2, 4), nrhs=rng.randint(1, 2), edge=edge, **optics)
    if kind == "precond_apply":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp32", "fp64"]), N=_log_int(rng, 100, 3000),
                    lmax=rng.randint(2, 4), nrhs=rng.choice([1, 1, 4]), edge=edge, **optics)
    if kind == "setup":
        beam = rng.choice(["gaussian", "plane"])
        return dict(kind=kind, beam=beam, N=_log_int(rng, 50, 10000), lmax=rng.randint(1, 5),
                    nrhs=1 if beam == "gaussian" else rng.randint(1, 8), **optics)
    if kind == "farfield":
        return dict(kind=kind, N=_log_int(rng, 50, 6000), lmax=rng.randint(2, 5), directions=_log_int(rng, 50, 3000),
                    **optics)
    if kind == "nearfield":
        return dict(kind=kind, beam=rng.choice(["gaussian", "plane"]), N=_log_int(rng, 20, 1000),
                    lmax=rng.randint(1, 5), points=_log_int(rng, 100, 5000), **optics)
    return dict(kind=kind, mode=rng.choice(["mixed", "fp64"]), solver=rng.choice(["gmres", "bicgstab"]),
                N=rng.randint(20, 130), lmax=rng.randint(1, 3), nrhs=rng.choice([1, 2]),
                edge=rng.choice([0.0, edge]), **optics)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed, part=0):
    return np.random.Generator(np.random.PCG64([int(seed), part]))


def _packing(gen, N, poly, slab):
    """Disjoint spheres on the jittered sites of a cubic lattice: a cube, or a slab 2 um (polydisperse) or 4 um
    thick.  Sites in random order, some of them vacant."""
    if poly:
        mu = math.log(150.0) - RADIUS_SIGMA ** 2 / 2.0
        radii = np.exp(np.clip(gen.normal(mu, RADIUS_SIGMA, N), mu - 3 * RADIUS_SIGMA, mu + 3 * RADIUS_SIGMA))
    else:
        radii = np.full(N, 130.0 if slab else 100.0)
    rmax = float(radii.max())
    a = 2.0 * rmax * 1.12
    if slab:
        nz = max(1, int((2000.0 if poly else 4000.0) / a))
        nx = max(1, math.ceil(math.sqrt(1.05 * N / nz)))
        shape = (nx, nx, nz)
    else:
        n = max(2, math.ceil((1.05 * N) ** (1.0 / 3.0)))
        shape = (n, n, n)
    sites = gen.permutation(shape[0] * shape[1] * shape[2])[:N]
    grid = np.stack(np.unravel_index(sites, shape), axis=1).astype(float)
    jitter = 0.999 * (a / 2.0 - rmax)
    pos = (grid + 0.5) * a + gen.uniform(-jitter, jitter, (N, 3))
    pos[:, :2] -= 0.5 * a * shape[0]
    return pos, radii


def _scene(case, seed):
    gen = _generator(seed)
    N = case["N"]
    slab = N >= 5000
    pos, radii = _packing(gen, N, case["poly"], slab)
    return pos, radii, np.full(N, complex(case["index_re"], case["index_im"])), gen


def _incidents(case, seed, nrhs):
    """Gaussian beam on the face of the packing, or plane waves within 60 degrees of the z axis."""
    if case.get("beam") == "gaussian":
        return [dict(kind="gaussian", waist=2000.0, focus=(30.0, -20.0, 0.0))] * nrhs
    gen = _generator(seed, 1)
    return [dict(kind="plane", beta=float(np.arccos(gen.uniform(0.5, 1.0))), alpha=float(gen.uniform(0, 2 * np.pi)),
                 pol=2 - (q % 2)) for q in range(nrhs)]


def _simulation(case, seed, incidents=0):
    pos, radii, index, gen = _scene(case, seed)
    sim = celes.Simulation(pos, radii, index, 1.0, case["wavelength"], case["lmax"])
    if incidents:
        binding.celes_set_incident(sim.ctx, [celes.make_incident(**d) for d in _incidents(case, seed, incidents)])
    return sim, gen


def _degrees(lmax):
    return np.array([l for _ in (1, 2) for l in range(1, lmax + 1) for _m in range(2 * l + 1)])


def _vector(seed, nrhs, N, lmax, precision):
    """Coefficient vectors: complex normal, smaller at higher degree as expansion coefficients are (host, FP64)."""
    gen = _generator(seed, 2)
    scale = 0.6 ** (_degrees(lmax) - 1.0)
    v = (gen.standard_normal((nrhs, N, scale.size)) + 1j * gen.standard_normal((nrhs, N, scale.size))) * scale
    return v.astype(np.complex64) if precision == "fp32" else v


def _prec(case):
    return celes.CELES_FP32 if case["precision"] == "fp32" else celes.CELES_FP64


def _ensembles(case, seed):
    """The batch's members: (case of one Simulation, its seed)."""
    gen = _generator(seed, 3)
    # sizes and degrees by the case alone, so that every seed is the same amount of work
    plan = _generator(case["ensembles"] * 1000 + case["n_hi"], 4)
    out = []
    for e in range(case["ensembles"]):
        out.append(dict(kind="ensemble", N=int(plan.integers(case["n_lo"], case["n_hi"] + 1)),
                        lmax=int(plan.integers(2, 6)), poly=False, wavelength=float(gen.uniform(400.0, 800.0)),
                        index_re=float(gen.uniform(1.45, 2.0)), index_im=0.0, seed=int(gen.integers(1 << 30))))
    return out


def _directions(case, seed):
    gen = _generator(seed, 5)
    n = case["directions"]
    return np.stack([np.arccos(gen.uniform(-1.0, 1.0, n)), gen.uniform(0.0, 2 * np.pi, n)], axis=1)


def _points(case, seed, pos):
    """Points of a plane x = const through the packing and a margin around it."""
    gen = _generator(seed, 6)
    n = case["points"]
    lo, hi = pos.min(axis=0) - 500.0, pos.max(axis=0) + 500.0
    p = gen.uniform(lo, hi, (n, 3))
    p[:, 0] = 0.25 * lo[0] + 0.75 * hi[0]
    return p


def _store_solution(sim, b):
    """Put b into the context as its solution: a user's guess, accepted as it is."""
    binding.celes_set_initial_guess(sim.ctx, b)
    binding.celes_solve(sim.ctx, 1e30, mode=celes.CELES_SOLVE_FP64, x0=celes.CELES_X0_USER, use_precond=False)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "setup":
        pos, radii, index, _ = _scene(case, seed)
        descs = [celes.make_incident(**d) for d in _incidents(case, seed, case["nrhs"])]
        return dict(kind=kind, args=(pos, radii, index, 1.0, case["wavelength"], case["lmax"]), descs=descs)
    if kind == "batch":
        sims, xs = [], []
        for m in _ensembles(case, seed):
            sim, _ = _simulation(m, m["seed"], incidents=case["rhs"])
            sims.append(sim)
            xs.append(_vector(m["seed"], case["rhs"], m["N"], m["lmax"], case["precision"]).reshape(-1))
        batch = celes.BatchSolver(sims)
        x = torch.from_numpy(np.concatenate(xs)).cuda()
        torch.cuda.synchronize()
        return dict(kind=kind, batch=batch, x=x, y=torch.empty_like(x), precision=_prec(case))
    if kind in ("matvec", "precond_build", "precond_apply"):
        sim, _ = _simulation(case, seed)
        x = torch.from_numpy(_vector(seed, case["nrhs"], case["N"], case["lmax"], case["precision"])).cuda()
        if kind == "precond_apply":
            sim.precond_build(case["edge"])
        torch.cuda.synchronize()
        return dict(kind=kind, op=case.get("op"), sim=sim, x=x, y=torch.empty_like(x), nrhs=case["nrhs"],
                    precision=_prec(case), edge=case.get("edge"), stream=torch.cuda.Stream())
    if kind == "solve":
        sim, _ = _simulation(case, seed, incidents=case["nrhs"])
        if case["edge"]:
            sim.precond_build(case["edge"])
        return dict(kind=kind, sim=sim, options=dict(
            mode=celes.CELES_SOLVE_MIXED if case["mode"] == "mixed" else celes.CELES_SOLVE_FP64,
            solver=celes.CELES_SOLVER_GMRES if case["solver"] == "gmres" else celes.CELES_SOLVER_BICGSTAB))
    sim, _ = _simulation(case, seed, incidents=1)
    _store_solution(sim, _vector(seed, 1, case["N"], case["lmax"], "fp64"))
    if kind == "farfield":
        return dict(kind=kind, sim=sim, dirs=_directions(case, seed))
    return dict(kind=kind, sim=sim, points=_points(case, seed, _scene(case, seed)[0]))


def run(state):
    kind = state["kind"]
    if kind == "matvec":
        call = binding.celes_coupling_matvec if state["op"] == "coupling" else binding.celes_master_matvec
        call(state["sim"].ctx, state["x"], state["y"], state["nrhs"], state["precision"], state["stream"])
        return state["y"]
    if kind == "batch":
        binding.celes_batch_master_matvec(state["batch"].b, state["x"], state["y"], state["precision"])
        return state["y"]
    if kind in ("precond_build", "precond_apply"):
        if kind == "precond_build":
            state["sim"].precond_build(state["edge"])
        binding.celes_precond_apply(state["sim"].ctx, state["x"], state["y"], state["nrhs"], state["precision"],
                                    state["stream"])
        return state["y"]
    if kind == "setup":
        sim = celes.Simulation(*state["args"])
        binding.celes_set_incident(sim.ctx, state["descs"])
        out = dict(tmatrix=sim.tmatrix(), incident=sim.incident_coefficients())
        sim.close()
        return out
    if kind == "farfield":
        return state["sim"].farfield(state["dirs"])
    if kind == "nearfield":
        return state["sim"].nearfield(state["points"])
    state["sim"].solve(1e-12, **state["options"])
    return state["sim"].coefficients()


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _pair_flops(lmax):
    """Two rotations (the cosine and sine blocks of every degree) and the axial products of one ordered pair."""
    rot = sum(2 * l * l + 2 * l + 1 for l in range(1, lmax + 1))
    axial = 2 * lmax * lmax + 4 * sum((lmax - mu + 1) ** 2 for mu in range(1, lmax + 1))
    return 16.0 * rot + 8.0 * axial


def _nmax(lmax):
    return 2 * lmax * (lmax + 2)


def _blocks(case, seed=0):
    """Unknowns of the preconditioner's blocks: spheres by the cuboid that holds their centre, cuboids in (z, y, x)
    order, counted from the minimum corner of the centres."""
    pos = _scene(case, seed)[0]
    cell = np.floor((pos - pos.min(axis=0)) / case["edge"]).astype(np.int64)
    order = np.lexsort((cell[:, 0], cell[:, 1], cell[:, 2]))
    cut = np.flatnonzero(np.any(np.diff(cell[order], axis=0) != 0, axis=1)) + 1
    return [b for b in np.split(order, cut)]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        elem = 8 if case["precision"] == "fp32" else 16
        members = _ensembles(case, 0)
        return {"bytes": sum(2.0 * case["rhs"] * m["N"] * _nmax(m["lmax"]) * elem + 32.0 * m["N"] for m in members),
                "flops": sum(case["rhs"] * m["N"] * (m["N"] - 1.0) * _pair_flops(m["lmax"]) for m in members)}
    N, L = case["N"], case["lmax"]
    nm = _nmax(L)
    if kind == "matvec":
        elem = 8 if case["precision"] == "fp32" else 16
        return {"bytes": 2.0 * case["nrhs"] * N * nm * elem + 32.0 * N,
                "flops": case["nrhs"] * N * (N - 1.0) * _pair_flops(L)}
    if kind in ("precond_build", "precond_apply"):
        elem = 8 if case["precision"] == "fp32" else 16
        dims = [float(len(b) * nm) for b in _blocks(case)]
        entries = sum(d * d for d in dims)
        vectors = 2.0 * case["nrhs"] * N * nm * elem
        if kind == "precond_apply":
            return {"bytes": entries * elem + vectors, "flops": 8.0 * case["nrhs"] * entries}
        return {"bytes": entries * 16 + entries * elem + vectors, "flops": sum(8.0 / 3.0 * d ** 3 for d in dims)}
    if kind == "setup":
        return {"bytes": 48.0 * N + 16.0 * N * nm * (1 + case["nrhs"]),
                "flops": case["nrhs"] * N * nm * 8.0 * (128 if case["beam"] == "gaussian" else 1)}
    if kind == "farfield":
        D = case["directions"]
        return {"bytes": 32.0 * N + 16.0 * N * nm + 48.0 * D, "flops": 8.0 * D * N * nm}
    if kind == "nearfield":
        return {"bytes": 32.0 * N + 16.0 * N * nm + 72.0 * case["points"], "flops": 24.0 * case["points"] * N * nm}
    return {"bytes": 32.0 * N * nm * case["nrhs"], "flops": 20.0 * case["nrhs"] * N * (N - 1.0) * _pair_flops(L)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch and numpy
# ---------------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


@lru_cache(maxsize=None)
def _w3j(j1, j2, j3, m1, m2, m3):
    """Wigner 3j symbol by Racah's formula in exact fractions."""
    if m1 + m2 + m3 or j3 < abs(j1 - j2) or j3 > j1 + j2 or abs(m1) > j1 or abs(m2) > j2 or abs(m3) > j3:
        return 0.0
    f = math.factorial
    delta = Fraction(f(j1 + j2 - j3) * f(j1 - j2 + j3) * f(j2 + j3 - j1), f(j1 + j2 + j3 + 1))
    pre = f(j1 + m1) * f(j1 - m1) * f(j2 + m2) * f(j2 - m2) * f(j3 + m3) * f(j3 - m3)
    s = Fraction(0)
    for k in range(max(0, j2 - j3 - m1, j1 - j3 + m2), min(j1 + j2 - j3, j1 - m1, j2 + m2) + 1):
        s += Fraction((-1) ** k, f(k) * f(j3 - j2 + k + m1) * f(j3 - j1 + k - m2) * f(j1 + j2 - j3 - k)
                      * f(j1 - k - m1) * f(j2 - k + m2))
    q = delta * pre * s * s
    return (-1.0) ** ((j1 - j2 - m3) % 2) * math.copysign(1.0, s) * math.sqrt(q.numerator / q.denominator) if s else 0.0


@lru_cache(maxsize=None)
def _ab5(l, m, lp, mp, p):
    """a5 and b5 of the addition theorem for vector spherical wave functions."""
    phase = 1j ** ((abs(m - mp) - abs(m) - abs(mp) + lp - l + p) % 4) * (-1.0) ** ((m - mp) % 2)
    common = math.sqrt((2 * l + 1) * (2 * lp + 1) / (2.0 * l * (l + 1) * lp * (lp + 1))) * _w3j(l, lp, p, m, -mp, mp - m)
    a = phase * (l * (l + 1) + lp * (lp + 1) - p * (p + 1)) * math.sqrt(2 * p + 1) * common * _w3j(l, lp, p, 0, 0, 0)
    b = 0.0
    prod = (l + lp + 1 + p) * (l + lp + 1 - p) * (p + l - lp) * (p - l + lp) * (2 * p + 1)
    if p >= 1 and prod > 0:
        b = phase * math.sqrt(prod) * common * _w3j(l, lp, p - 1, 0, 0, 0)
    return complex(a), complex(b)


@lru_cache(maxsize=None)
def _coupling_table(lmax):
    """For every q = m' - m: entries (receiving row, source row) and the real matrices that take (Re, Im) of
    h_p P_p^|q| to (Re, Im) of A + B and of A - B."""
    rows = [(l, m) for l in range(1, lmax + 1) for m in range(-l, l + 1)]
    out = []
    for q in range(-2 * lmax, 2 * lmax + 1):
        ps = list(range(abs(q), 2 * lmax + 1))
        pairs = [(ro, ri) for ro, (l, m) in enumerate(rows) for ri, (lp, mp) in enumerate(rows) if mp - m == q]
        a, b = np.zeros((len(ps), len(pairs))), np.zeros((len(ps), len(pairs)))
        for e, (ro, ri) in enumerate(pairs):
            (l, m), (lp, mp) = rows[ro], rows[ri]
            for k, p in enumerate(ps):
                if abs(l - lp) <= p <= l + lp:
                    a5, b5 = _ab5(lp, mp, l, m, p)
                    a[k, e], b[k, e] = a5.real, b5.imag
        # (A + B) = (Sr + i Si)(a + i b): Re = Sr a - Si b, Im = Si a + Sr b
        plus = np.block([[a, b], [-b, a]])
        minus = np.block([[a, -b], [b, a]])
        out.append((q, [e[0] for e in pairs], [e[1] for e in pairs], plus, minus))
    return out


def _hankel(pmax, x):
    """h_p(x), p = 0..pmax: closed forms of the first two and upward recurrence."""
    e = torch.polar(torch.ones_like(x), x)
    h = [-1j * e / x, e * (-1.0 / x - 1j / (x * x))]
    for p in range(1, pmax):
        h.append((2 * p + 1) / x * h[p] - h[p - 1])
    return h[: pmax + 1]


def _legendre(lmax, ct, st):
    """Normalised associated Legendre functions P[l][m] (no Condon-Shortley phase)."""
    P = [[None] * (l + 1) for l in range(lmax + 1)]
    d = torch.full_like(ct, math.sqrt(0.5))
    for m in range(lmax + 1):
        if m:
            d = d * (math.sqrt((2 * m + 1.0) / (2 * m)) * st)
        P[m][m] = d
        if m < lmax:
            P[m + 1][m] = math.sqrt(2 * m + 3.0) * ct * d
        for l in range(m + 2, lmax + 1):
            a = math.sqrt((4.0 * l * l - 1) / (l * l - m * m))
            b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1) ** 2 - 1))
            P[l][m] = a * (ct * P[l - 1][m] - b * P[l - 2][m])
    return P


def _pair_terms(lmax, k, d):
    """Geometry of the separations d (.., 3): h_p P_p^mu and e^{i phi}."""
    r = torch.sqrt((d * d).sum(-1))
    rho = torch.hypot(d[..., 0], d[..., 1])
    P = _legendre(2 * lmax, d[..., 2] / r, rho / r)
    h = _hankel(2 * lmax, k * r)
    one = torch.where(rho > 0, rho, torch.ones_like(rho))
    ephi = torch.complex(torch.where(rho > 0, d[..., 0] / one, torch.ones_like(rho)), d[..., 1] / one)
    return h, P, ephi


def _exact_coupling(pos, k, lmax, x):
    """y_i = sum over j != i of W_ij x_j; x (nrhs, N, nmax)."""
    dev = _device()
    p = torch.as_tensor(pos, device=dev)
    x = torch.as_tensor(np.asarray(x, dtype=np.complex128), device=dev)
    N, NH = p.shape[0], lmax * (lmax + 2)
    xs = (x[..., :NH] + x[..., NH:], x[..., :NH] - x[..., NH:])
    ys = [torch.zeros(x.shape[0], N, NH, dtype=torch.complex128, device=dev) for _ in (0, 1)]
    table = [(q, torch.tensor(ro, device=dev), torch.tensor(ri, device=dev),
              (torch.as_tensor(plus, device=dev), torch.as_tensor(minus, device=dev)))
             for q, ro, ri, plus, minus in _coupling_table(lmax)]
    step = max(1, int((2.0e9 if dev.type == "cuda" else 5e7) / (N * NH * 64)))
    eye = torch.arange(N, device=dev)
    for i0 in range(0, N, step):
        i1 = min(N, i0 + step)
        d = p[i0:i1, None, :] - p[None, :, :]
        self_ = eye[i0:i1, None] == eye[None, :]
        d = torch.where(self_[..., None], torch.ones_like(d), d)
        h, P, ephi = _pair_terms(lmax, k, d)
        for q, ro, ri, mats in table:
            m = abs(q)
            s = torch.stack([h[t] * P[t][m] for t in range(m, 2 * lmax + 1)], dim=-1)
            s = s * torch.where(self_, torch.zeros_like(ephi), (ephi if q >= 0 else ephi.conj()) ** m)[..., None]
            s = torch.cat([s.real, s.imag], dim=-1)
            for sign in (0, 1):
                g = s @ mats[sign]
                n = g.shape[-1] // 2
                for r in range(x.shape[0]):
                    xe = xs[sign][r][:, ri]
                    gr, gi = g[..., :n], g[..., n:]
                    re = (gr * xe.real).sum(1) - (gi * xe.imag).sum(1)
                    im = (gr * xe.imag).sum(1) + (gi * xe.real).sum(1)
                    ys[sign][r, i0:i1].index_add_(1, ro, torch.complex(re, im))
    return torch.cat([(ys[0] + ys[1]) / 2, (ys[0] - ys[1]) / 2], dim=-1)


def _exact_block(pos, k, lmax):
    """Dense W (n nmax, n nmax) of a few spheres, zero on the diagonal blocks."""
    dev = _device()
    p = torch.as_tensor(pos, device=dev)
    n, NH = p.shape[0], lmax * (lmax + 2)
    d = p[:, None, :] - p[None, :, :]
    self_ = torch.eye(n, dtype=torch.bool, device=dev)
    d = torch.where(self_[..., None], torch.ones_like(d), d)
    h, P, ephi = _pair_terms(lmax, k, d)
    W = torch.zeros(n, n, 2, NH, 2, NH, dtype=torch.complex128, device=dev)
    for q, ro, ri, plus, minus in _coupling_table(lmax):
        m = abs(q)
        s = torch.stack([h[t] * P[t][m] for t in range(m, 2 * lmax + 1)], dim=-1)
        s = s * torch.where(self_, torch.zeros_like(ephi), (ephi if q >= 0 else ephi.conj()) ** m)[..., None]
        s = torch.cat([s.real, s.imag], dim=-1)
        g = [s @ torch.as_tensor(v, device=dev) for v in (plus, minus)]
        g = [torch.complex(v[..., : v.shape[-1] // 2], v[..., v.shape[-1] // 2:]) for v in g]
        A, B = (g[0] + g[1]) / 2, (g[0] - g[1]) / 2
        W[:, :, 0, ro, 0, ri] = A
        W[:, :, 1, ro, 1, ri] = A
        W[:, :, 0, ro, 1, ri] = B
        W[:, :, 1, ro, 0, ri] = B
    return W.reshape(n, n, 2 * NH, 2 * NH).permute(0, 2, 1, 3).reshape(n * 2 * NH, n * 2 * NH)


def _bessel_j(lmax, z):
    """Spherical Bessel functions j_0..j_lmax by downward recurrence."""
    z = np.asarray(z, dtype=complex)
    top = lmax + 40 + int(2 * np.max(np.abs(z)))
    up, cur = np.zeros_like(z), np.full_like(z, 1e-200)
    out = [None] * (lmax + 1)
    for l in range(top, 0, -1):
        up, cur = cur, (2 * l + 1) / z * cur - up
        if l <= lmax + 1:
            out[l - 1] = cur
        big = np.abs(cur) > 1e100
        if np.any(big):
            f = np.where(big, 1e-100, 1.0)
            up, cur = up * f, cur * f
            out = [None if o is None else o * f for o in out]
    j0, j1 = np.sin(z) / z, np.sin(z) / z ** 2 - np.cos(z) / z
    use0 = np.abs(j0) >= np.abs(j1)
    scale = np.where(use0, j0 / out[0], j1 / out[1])
    return [o * scale for o in out]


def _exact_t(lmax, k, radii, n_rel):
    """Diagonal of T, (N, nmax)."""
    x = k * np.asarray(radii)
    y = n_rel * x
    jx, jy = [v.real for v in _bessel_j(lmax, x)], _bessel_j(lmax, y)
    yx = [-np.cos(x) / x, -np.cos(x) / x ** 2 - np.sin(x) / x]
    for l in range(1, lmax):
        yx.append((2 * l + 1) / x * yx[l] - yx[l - 1])
    q = ([], [])
    for l in range(1, lmax + 1):
        h, hm = jx[l] + 1j * yx[l], jx[l - 1] + 1j * yx[l - 1]
        djx, djy, dhx = x * jx[l - 1] - l * jx[l], y * jy[l - 1] - l * jy[l], x * hm - l * h
        m2 = n_rel ** 2
        q[0].append((jx[l] * djy - jy[l] * djx) / (jy[l] * dhx - h * djy))
        q[1].append((jx[l] * djy - m2 * jy[l] * djx) / (m2 * jy[l] * dhx - h * djy))
    return np.stack([q[t][l - 1] for t in (0, 1) for l in range(1, lmax + 1) for _ in range(2 * l + 1)], axis=1)


def _pi_tau(lmax, ct, st):
    """pi[l][m] = P/sin and tau[l][m] = dP/dtheta, valid at sin = 0 too."""
    # Q[l][m] = P_l^m / sin^m by the recursion in l; pi = Q sin^(m-1)
    Q = _legendre(lmax + 1, ct, torch.ones_like(st))
    power = [torch.ones_like(st)]
    for _ in range(lmax + 1):
        power.append(power[-1] * st)
    P = [[Q[l][m] * power[m] for m in range(l + 1)] for l in range(lmax + 1)]
    pi = [[torch.zeros_like(ct) if m == 0 else Q[l][m] * power[m - 1] for m in range(l + 1)] for l in range(lmax + 1)]
    tau = [[None] * (l + 1) for l in range(lmax + 1)]
    for l in range(1, lmax + 1):
        for m in range(l + 1):
            if m == 0:
                tau[l][0] = -math.sqrt(l * (l + 1.0)) * pi[l][1] * st
            else:
                prev = pi[l - 1][m] if m <= l - 1 else torch.zeros_like(ct)
                tau[l][m] = l * ct * pi[l][m] - math.sqrt((2 * l + 1.0) * (l * l - m * m) / (2 * l - 1.0)) * prev
    return P, pi, tau


def _b_transform(lmax, beta, dagger):
    """B_nj(beta): dict (tau, l, m, j) -> tensor shaped like beta."""
    _, pi, tau = _pi_tau(lmax, torch.cos(beta), torch.sin(beta))
    iu = -1j if dagger else 1j
    return {(t, l, m, j): -1.0 / iu ** (l + 1) / math.sqrt(2.0 * l * (l + 1)) * (iu if j == 1 else 1.0)
            * (tau[l][abs(m)] if t == j else m * pi[l][abs(m)])
            for t in (1, 2) for l in range(1, lmax + 1) for m in range(-l, l + 1) for j in (1, 2)}


def _rows(lmax):
    return [(t, l, m) for t in (1, 2) for l in range(1, lmax + 1) for m in range(-l, l + 1)]


def _beam_nodes(k, w, count=200):
    s2 = 39.2 / ((w * k) ** 2 / 4.0)
    top = math.pi / 2 if s2 >= 1.0 else math.asin(math.sqrt(s2))
    x, g = np.polynomial.legendre.leggauss(count)
    dev = _device()
    beta = torch.as_tensor(0.5 * top * (x + 1.0), device=dev)
    weight = torch.as_tensor(0.5 * top * g, device=dev)
    sb, cb = torch.sin(beta), torch.cos(beta)
    return beta, sb, cb, weight * sb * cb * torch.exp(-(w * k * sb) ** 2 / 4.0)


def _exact_incident(case, seed, pos, k):
    """a_in (nrhs, N, nmax)."""
    dev, L = _device(), case["lmax"]
    p = torch.as_tensor(pos, device=dev)
    out = []
    for inc in _incidents(case, seed, case["nrhs"]):
        a = torch.zeros(p.shape[0], _nmax(L), dtype=torch.complex128, device=dev)
        if inc["kind"] == "plane":
            be, al = inc["beta"], inc["alpha"]
            kv = k * torch.tensor([math.sin(be) * math.cos(al), math.sin(be) * math.sin(al), math.cos(be)],
                                  dtype=torch.float64, device=dev)
            e = torch.polar(torch.ones(p.shape[0], dtype=torch.float64, device=dev), p @ kv)
            B = _b_transform(L, torch.tensor([be], dtype=torch.float64, device=dev), True)
            for n, (t, l, m) in enumerate(_rows(L)):
                a[:, n] = 4.0 * e * np.exp(-1j * m * al) * B[t, l, m, inc["pol"]][0]
        else:
            w, aG = inc["waist"], -math.pi / 2
            rel = p - torch.tensor(inc["focus"], dtype=torch.float64, device=dev)
            rho, phi = torch.hypot(rel[:, 0], rel[:, 1]), torch.atan2(rel[:, 1], rel[:, 0])
            beta, sb, cb, gw = _beam_nodes(k, w)
            B = _b_transform(L, beta, True)
            na = int(k * float(rho.max()) * float(sb.max()) + 3 * L + 60)
            al = math.pi * (torch.arange(na, dtype=torch.float64, device=dev) + 0.5) / na
            cosm = torch.stack([torch.cos(m * al) for m in range(L + 2)], dim=1).to(torch.complex128) / na
            step = max(1, int(2e8 / (na * beta.numel())) if dev.type == "cuda" else 4)
            for i0 in range(0, p.shape[0], step):
                i1 = min(p.shape[0], i0 + step)
                arg = (k * rho[i0:i1, None] * sb[None, :])[..., None] * torch.cos(al)
                bes = torch.polar(torch.ones_like(arg), arg) @ cosm  # i^m J_m
                z = torch.polar(gw[None, :].expand(i1 - i0, -1).contiguous(), k * rel[i0:i1, 2, None] * cb[None, :])

                def M(m):
                    return 2.0 * math.pi * torch.polar(torch.ones_like(phi[i0:i1]), -m * phi[i0:i1])[:, None] \
                        * bes[..., abs(m)]

                for n, (t, l, m) in enumerate(_rows(L)):
                    u, v = np.exp(-1j * aG) * M(m - 1), np.exp(1j * aG) * M(m + 1)
                    f = B[t, l, m, 1] * (u + v) / 2 + B[t, l, m, 2] * (-1j * u + 1j * v) / 2
                    a[i0:i1, n] = (k * w) ** 2 / math.pi * (z * f).sum(1)
        out.append(a)
    return torch.stack(out)


def _exact_farfield(pos, k, L, b, dirs):
    dev = _device()
    p, b = torch.as_tensor(pos, device=dev), torch.as_tensor(b, device=dev)
    d = torch.as_tensor(dirs, device=dev)
    B = _b_transform(L, d[:, 0], False)
    kv = k * torch.stack([torch.sin(d[:, 0]) * torch.cos(d[:, 1]), torch.sin(d[:, 0]) * torch.sin(d[:, 1]),
                          torch.cos(d[:, 0])], dim=1)
    out = torch.zeros(d.shape[0], 2, dtype=torch.complex128, device=dev)
    step = max(1, int(2e8 / p.shape[0]))
    for q in range(0, d.shape[0], step):
        ph = -(kv[q:q + step] @ p.T)
        s = torch.polar(torch.ones_like(ph), ph) @ b
        for n, (t, l, m) in enumerate(_rows(L)):
            e = torch.polar(torch.ones_like(d[q:q + step, 1]), m * d[q:q + step, 1])
            for j in (1, 2):
                out[q:q + step, j - 1] += B[t, l, m, j][q:q + step] * e * s[:, n] / (2.0 * math.pi)
    return out


def _exact_nearfield(case, seed, pos, radii, k, b, pts):
    """Scattered plus incident field, NaN inside a sphere."""
    dev, L = _device(), case["lmax"]
    NH = L * (L + 2)
    p, R = torch.as_tensor(pos, device=dev), torch.as_tensor(radii, device=dev)
    b, r = torch.as_tensor(b, device=dev), torch.as_tensor(pts, device=dev)
    E = torch.zeros(r.shape[0], 3, dtype=torch.complex128, device=dev)
    inside = torch.zeros(r.shape[0], dtype=torch.bool, device=dev)
    step = max(1, int((2e7 if dev.type == "cuda" else 1e5) / p.shape[0]))
    for q in range(0, r.shape[0], step):
        d = r[q:q + step, None, :] - p[None]
        dist = torch.sqrt((d * d).sum(-1))
        inside[q:q + step] = (dist < R).any(1)
        rho = torch.hypot(d[..., 0], d[..., 1])
        ct, st = d[..., 2] / dist, rho / dist
        one = torch.where(rho > 0, rho, torch.ones_like(rho))
        cp, sp = torch.where(rho > 0, d[..., 0] / one, torch.ones_like(rho)), d[..., 1] / one
        x = k * dist
        h = _hankel(L, x)
        P, pi, tau = _pi_tau(L, ct, st)
        Er, Et, Ep = (torch.zeros(d.shape[:2], dtype=torch.complex128, device=dev) for _ in range(3))
        for l in range(1, L + 1):
            dxh = h[l - 1] - l / x * h[l]
            for m in range(-l, l + 1):
                e = torch.complex(cp, sp if m >= 0 else -sp) ** abs(m) / math.sqrt(2.0 * l * (l + 1))
                row = l * (l + 1) - 1 + m
                c1, c2 = b[:, row] * e, b[:, NH + row] * e
                am = abs(m)
                Er += c2 * l * (l + 1) * h[l] / x * P[l][am]
                Et += c1 * h[l] * 1j * m * pi[l][am] + c2 * dxh * tau[l][am]
                Ep += -c1 * h[l] * tau[l][am] + c2 * dxh * 1j * m * pi[l][am]
        E[q:q + step, 0] = (st * cp * Er + ct * cp * Et - sp * Ep).sum(1)
        E[q:q + step, 1] = (st * sp * Er + ct * sp * Et + cp * Ep).sum(1)
        E[q:q + step, 2] = (ct * Er - st * Et).sum(1)
    inc = _incidents(case, seed, 1)[0]
    if inc["kind"] == "plane":
        be, al = inc["beta"], inc["alpha"]
        kv = k * torch.tensor([math.sin(be) * math.cos(al), math.sin(be) * math.sin(al), math.cos(be)],
                              dtype=torch.float64, device=dev)
        vec = [-math.sin(al), math.cos(al), 0.0] if inc["pol"] == 1 else \
            [math.cos(be) * math.cos(al), math.cos(be) * math.sin(al), -math.sin(be)]
        ph = r @ kv
        E += torch.polar(torch.ones_like(ph), ph)[:, None] * torch.tensor(vec, dtype=torch.float64, device=dev)
    else:
        w, aG = inc["waist"], -math.pi / 2
        rel = r - torch.tensor(inc["focus"], dtype=torch.float64, device=dev)
        _, sb, cb, gw = _beam_nodes(k, w)
        na = 2 * (int(k * float(torch.hypot(rel[:, 0], rel[:, 1]).max())) + 40)
        al = 2.0 * math.pi * torch.arange(na, dtype=torch.float64, device=dev) / na
        ca, sa = torch.cos(al), torch.sin(al)
        cd, sd = torch.cos(al - aG), torch.sin(al - aG)
        amp = (k * w) ** 2 / (4.0 * math.pi) * 2.0 * math.pi / na
        for s, c, g in zip(sb.tolist(), cb.tolist(), gw.tolist()):
            vec = torch.stack([-cd * sa + sd * c * ca, cd * ca + sd * c * sa, -sd * s], dim=1)
            ph = k * (s * (rel[:, :1] * ca + rel[:, 1:2] * sa) + c * rel[:, 2:3])
            E += amp * g * (torch.polar(torch.ones_like(ph), ph) @ vec.to(torch.complex128))
    E[inside] = complex(float("nan"), float("nan"))
    return E


#: products of pairs and matrix entries that plain torch does in about ten seconds on a GPU
MOST_ENTRIES = 7e10


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _ensembles(case, seed)
        if case["rhs"] * sum(m["N"] ** 2 * (m["lmax"] * (m["lmax"] + 2)) ** 2 for m in members) > MOST_ENTRIES:
            return None
        out = []
        for m in members:
            pos, radii, index, _ = _scene(m, m["seed"])
            k = 2.0 * math.pi / m["wavelength"]
            x = _vector(m["seed"], case["rhs"], m["N"], m["lmax"], case["precision"]).astype(np.complex128)
            y = _exact_coupling(pos, k, m["lmax"], x).cpu().numpy()
            out.append((x - _exact_t(m["lmax"], k, radii, index)[None] * y).reshape(-1))
        return np.concatenate(out)
    N, L = case["N"], case["lmax"]
    pos, radii, index, _ = _scene(case, seed)
    k = 2.0 * math.pi / case["wavelength"]
    if kind == "matvec":
        if (1 + case["nrhs"]) * 0.5 * N ** 2 * (L * (L + 2)) ** 2 > MOST_ENTRIES:
            return None
        x = _vector(seed, case["nrhs"], N, L, case["precision"]).astype(np.complex128)
        y = _exact_coupling(pos, k, L, x).cpu().numpy()
        return y if case["op"] == "coupling" else x - _exact_t(L, k, radii, index)[None] * y
    if kind in ("precond_build", "precond_apply"):
        x = _vector(seed, case["nrhs"], N, L, case["precision"]).astype(np.complex128)
        T = _exact_t(L, k, radii, index)
        y = np.empty_like(x)
        for b in _blocks(case, seed):
            M = torch.eye(len(b) * _nmax(L), dtype=torch.complex128, device=_device()) \
                - torch.as_tensor(T[b].reshape(-1, 1), device=_device()) * _exact_block(pos[b], k, L)
            rhs = torch.as_tensor(x[:, b].reshape(case["nrhs"], -1).T.copy(), device=_device())
            y[:, b] = torch.linalg.solve(M, rhs).T.reshape(case["nrhs"], len(b), -1).cpu().numpy()
        return y
    if kind == "setup":
        return dict(tmatrix=_exact_t(L, k, radii, index),
                    incident=_exact_incident(case, seed, pos, k).cpu().numpy())
    if kind == "solve":
        T = torch.as_tensor(_exact_t(L, k, radii, index), device=_device())
        M = torch.eye(N * _nmax(L), dtype=torch.complex128, device=_device()) \
            - T.reshape(-1, 1) * _exact_block(pos, k, L)
        rhs = (T[None] * _exact_incident(case, seed, pos, k)).reshape(case["nrhs"], -1).T
        return torch.linalg.solve(M, rhs).T.reshape(case["nrhs"], N, -1).cpu().numpy()
    b = _vector(seed, 1, N, L, "fp64")[0]
    if kind == "farfield":
        return _exact_farfield(pos, k, L, b, _directions(case, seed)).cpu().numpy()
    return _exact_nearfield(case, seed, pos, radii, k, b, _points(case, seed, pos)).cpu().numpy()
