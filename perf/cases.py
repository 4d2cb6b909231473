"""The work a user of this package gives it, as cases that can be timed and compared.

A calculation has four parts, each with its own public entry point: the matrix elements S and H at positions
of a projectile path (``Basis.matrix_elements``), the batched complex solve (``solve``), the propagation of the
amplitudes along many paths (``Basis.propagate``, and ``Batch`` for several bases in one launch), and the
gradient of the final probabilities (``Basis.propagate_adjoint``).  The sizes are those of the named workloads
(one-centre p + H with N = 59, two-centre p + H with N = 380, the velocity scan with N = 316 to 572, C6+ + H
with N = 1622, the p + Li-like gradient with N = 379), cut to a window of RK4 steps around closest approach
where a whole path would take minutes.

``exact`` restates the method in plain numpy FP64 from the generated inputs alone.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

import paper_2403_04252_gb300 as w
import wpccc_inputs as wi

SOLVES = {"stage": w.SOLVE_STAGE, "matrix": w.SOLVE_MATRIX, "schur": w.SOLVE_SCHUR}


def listed():
    p_h = dict(Z_P=1.0, nmax=4, lmax=3, nbins=10, kmax=3.0, nmax_P=4, lmax_P=3, nbins_P=10, Geta=48, Gtau=48, v=1.5)
    return [
        # the smallest call: elements of a one-centre basis (N = 59) at three positions, for a look at a potential
        # curve or a custom integrator that steps by itself; launches and the host path count
        dict(name="elements_1c_N59", kind="elements", centres=1, Z_P=1.0, nmax=3, lmax=2, nbins=5, kmax=2.0,
             v=1.0, positions=3, b_lo=0.5, b_hi=8.0, mode=0),
        # two-centre elements in plain FP64 at an odd number of positions (a z-scan of the couplings)
        dict(p_h, name="elements_2c_fp64_N380", kind="elements", centres=2, positions=21, b_lo=0.2, b_hi=12.0, mode=0),
        # the same with the reduced-precision tensor-core elements, on the largest velocity-scan basis (N = 572)
        dict(p_h, name="elements_2c_tc_N572", kind="elements", centres=2, nbins=16, nbins_P=16, Geta=72, v=4.0,
             positions=45, b_lo=0.2, b_hi=12.0, mode=3),
        # the paper's solve, S X = H by pivoted LU with N right-hand sides, for one position of each of 24 paths
        dict(name="solve_N380", kind="solve", N=380, batch=24),
        # whole one-centre paths: 8 impact parameters, z from -40 to 40 in 800 steps, from the ground state
        dict(name="propagate_1c_N59", kind="propagate", centres=1, Z_P=1.0, nmax=3, lmax=2, nbins=5, kmax=2.0, v=1.0,
             paths=8, steps=800, h=0.1, ragged=False, b_lo=0.5, b_hi=8.0, mode=0, solve="stage", iters=2),
        # a first look with the library's defaults (FP64, LU of S applied per RK4 stage): uneven centres, a node
        # count that is no multiple of 128, paths of different lengths
        dict(name="propagate_2c_default_N109", kind="propagate", centres=2, Z_P=1.0, nmax=3, lmax=2, nbins=5, kmax=2.0,
             nmax_P=3, lmax_P=2, nbins_P=4, Geta=50, Gtau=30, v=1.2, paths=5, steps=23, h=0.1, ragged=True,
             b_lo=0.5, b_hi=8.0, mode=0, solve="stage", iters=2),
        # the two-centre p + H workload in plain FP64 with the Schur solve: a window of all 32 paths
        dict(p_h, name="propagate_2c_fp64_N380", kind="propagate", centres=2, paths=32, steps=10, h=0.1, ragged=False,
             b_lo=0.2, b_hi=12.0, mode=0, solve="schur", iters=2),
        # the same at the FP64 bar on the tensor cores (mode 5 with four refinement sweeps)
        dict(p_h, name="propagate_2c_mode5_N380", kind="propagate", centres=2, paths=32, steps=16, h=0.1, ragged=False,
             b_lo=0.2, b_hi=12.0, mode=5, solve="schur", iters=4),
        # and in the fastest form within 1e-6 (mode 3), the one the benchmark reports
        dict(p_h, name="propagate_2c_mode3_N380", kind="propagate", centres=2, paths=32, steps=16, h=0.1, ragged=False,
             b_lo=0.2, b_hi=12.0, mode=3, solve="schur", iters=2),
        # bare C6+ on H, the largest basis (N = 1622) on its 128 x 48 rule, 16 paths near closest approach
        dict(name="propagate_C6_mode3_N1622", kind="propagate", centres=2, Z_P=6.0, nmax=6, lmax=5, nbins=20, kmax=4.0,
             nmax_P=6, lmax_P=5, nbins_P=20, Geta=128, Gtau=48, v=2.0, paths=16, steps=4, h=0.002, ragged=False,
             b_lo=0.5, b_hi=15.0, mode=3, solve="schur", iters=2),
        # the velocity scan: bases of uneven size and paths of uneven step count in one graph launch
        dict(name="batch_scan_mode3", kind="batch", speeds="0.5,1.2,4.0", paths=16, extent=1.6, b_lo=0.5, b_hi=12.0,
             mode=3),
        # gradients of capture and excitation for the Li-like target (FP64, checkpointed adjoint)
        dict(name="gradient_pLi_N379", kind="gradient", nmax=4, lmax=3, nbins=10, kmax=3.0, Geta=48, Gtau=48, v=1.5,
             paths=6, steps=4, h=0.1, checkpoint=2, b_lo=0.2, b_hi=12.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _states(nmax, lmax, nbins):
    return sum((2 * l + 1) * (max(0, nmax - l) + nbins) for l in range(lmax + 1))


def draw(rng):
    """One more case: the kind, the basis, the numbers of positions, paths and steps, the precision mode and the
    solve are drawn; the counts are cut so that the case stays below the largest listed ones."""
    kind = rng.choice(["elements"] * 3 + ["propagate"] * 5 + ["solve"] + ["batch"] + ["gradient"])
    if kind == "solve":
        N = _log(rng, 24, 600)
        return dict(kind="solve", N=N, batch=max(1, min(_log(rng, 1, 64), int(2.0e9 / N ** 3))))
    if kind == "batch":
        speeds = rng.sample([0.8, 1.2, 2.0, 3.0, 4.0], rng.randint(2, 3))
        return dict(kind="batch", speeds=",".join(str(s) for s in sorted(speeds)), paths=_log(rng, 2, 16),
                    extent=round(rng.uniform(0.8, 1.6), 3), b_lo=0.5, b_hi=12.0, mode=rng.choice([0, 3, 3, 5]))
    if kind == "gradient":
        return dict(kind="gradient", nmax=rng.randint(2, 4), lmax=rng.randint(1, 3), nbins=rng.randint(3, 10), kmax=3.0,
                    Geta=48, Gtau=rng.choice([32, 40, 48]), v=1.5, paths=_log(rng, 1, 6), steps=rng.randint(2, 4),
                    h=0.1, checkpoint=rng.randint(1, 4), b_lo=0.2, b_hi=12.0)
    centres = rng.choice([1, 2, 2, 2])
    if centres == 1:
        lmax = rng.randint(1, 5)
        case = dict(kind=kind, centres=1, Z_P=1.0, nmax=rng.randint(lmax + 1, 6), lmax=lmax, nbins=rng.randint(3, 20),
                    kmax=2.0, v=round(rng.uniform(1.0, 2.0), 3), b_lo=0.5, b_hi=8.0, mode=0)
        N = _states(case["nmax"], lmax, case["nbins"])
        cost = 60e-6 * (N / 380.0) ** 2
    else:
        # both centres l <= 3; node counts with and without a factor of 128
        Geta, Gtau = rng.choice([(48, 48), (48, 48), (72, 48), (64, 32), (50, 30), (60, 37)])
        case = dict(kind=kind, centres=2, Z_P=1.0, nmax=rng.randint(2, 4), lmax=rng.randint(1, 3),
                    nbins=rng.randint(3, 16), kmax=round(rng.uniform(2.0, 3.0), 2), nmax_P=rng.randint(2, 4),
                    lmax_P=rng.randint(1, 3), nbins_P=rng.randint(3, 16), Geta=Geta, Gtau=Gtau,
                    v=round(rng.uniform(1.2, 3.0), 3), b_lo=0.5, b_hi=12.0)
        NT = _states(case["nmax"], case["lmax"], case["nbins"])
        NP = _states(case["nmax_P"], case["lmax_P"], case["nbins_P"])
        N = NT + NP
        tensor = Geta * Gtau % 128 == 0
        case["mode"] = rng.choice(([0, 0, 3, 4] if tensor else [0, 0, 1]) if kind == "elements"
                                  else ([0, 0, 0, 3, 3, 4, 5] if tensor else [0, 0, 1, 2]))
        cost = NT * NP * Geta * Gtau * 12 / 1.2e12 + 4 * N ** 3 / 1e12
    if kind == "elements":
        case["positions"] = max(1, min(_log(rng, 1, 64), int(0.1 / cost)))
        return case
    paths = _log(rng, 1, 32)
    # (positions) x (assembly and solve) plus the serial stages of the sweep
    per_step = 2 * paths * cost + 4 * 0.5e-3 * max(0.05, (N / 380.0) ** 2)
    steps = max(2, min(_log(rng, 2, 400 if centres == 1 else 40), int(0.2 / per_step)))
    case.update(paths=paths, steps=steps, h=0.1, ragged=rng.random() < 0.5,
                solve=rng.choice(["schur", "schur", "stage", "matrix"]) if centres == 2 else "stage",
                iters=rng.choice([2, 2, 3, 4]))
    if case["mode"] in (1, 2, 3, 5) and case["solve"] == "matrix":
        case["solve"] = "schur"
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


@lru_cache(maxsize=None)
def _centre(Z, nmax, lmax, nbins, kmax):
    return wi.make_centre(Z, nmax, lmax, nbins, kmax, wi.radial_grid())


@lru_cache(maxsize=None)
def _li(nmax, lmax, nbins, kmax, Geta, Gtau):
    a, b = wi.li_parameters(0)
    return wi.li_basis(Z_p=1.0, a=a, b=b, nmax=nmax, lmax=lmax, nbins=nbins, kmax=kmax, Geta=Geta, Gtau=Gtau)


def _basis(case):
    """The basis a user's program keeps: hydrogenic states and wave packets on one or two centres."""
    if case["kind"] == "gradient":
        return _li(*(case[k] for k in ("nmax", "lmax", "nbins", "kmax", "Geta", "Gtau")))
    T = _centre(1.0, case["nmax"], case["lmax"], case["nbins"], case["kmax"])
    P = quad = None
    if case["centres"] == 2:
        P = _centre(case["Z_P"], case["nmax_P"], case["lmax_P"], case["nbins_P"], case["kmax"])
        quad = wi.make_quadrature(case["Geta"], case["Gtau"])
    return wi.Basis(grid=wi.radial_grid(), T=T, P=P, quad=quad, Z_T=1.0, Z_P=float(case["Z_P"]))


def _scan_case(case, v):
    """One speed of the velocity scan: packets per l and step length scale with v, 72 x 48 nodes."""
    nb = int(round(8 + 8 * (v - 0.5) / 3.5))
    h = 0.1 * v / 1.5
    return dict(kind="propagate", centres=2, Z_P=1.0, nmax=4, lmax=3, nbins=nb, kmax=3.0, nmax_P=4, lmax_P=3, nbins_P=nb,
                Geta=72, Gtau=48, v=v, paths=case["paths"], steps=max(1, int(round(case["extent"] / h))), h=h,
                ragged=False, b_lo=case["b_lo"], b_hi=case["b_hi"], mode=case["mode"], solve="schur", iters=2)


def _paths(case, rng):
    """b, v and z nodes of every path, and the amplitudes at its first node.  Whole paths start far out in the
    ground state; a window around closest approach starts in a spread-out mid-collision state."""
    n, steps, h = case["paths"], case["steps"], case["h"]
    b = np.sort(rng.uniform(case["b_lo"], case["b_hi"], n))
    v = case["v"] * (1.0 + 0.03 * rng.uniform(-1.0, 1.0))
    z0 = -0.5 * steps * h + 0.2 * h * rng.uniform(-1.0, 1.0)
    count = [steps if not case.get("ragged") else int(rng.integers(max(1, steps // 2), steps + 1)) for _ in range(n)]
    return b, v, [z0 + h * np.arange(k + 1, dtype=np.float64) for k in count]


def _amplitudes(case, rng, n, N):
    c = np.zeros((n, N), dtype=np.complex128)
    c[:, 0] = 1.0
    if case["steps"] * case["h"] < 60.0:
        d = rng.standard_normal((n, N)) + 1j * rng.standard_normal((n, N))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        c = 0.9 * c + 0.4 * d
    return c


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "solve":
        # an overlap-like matrix (identity plus decaying couplings, Hermitian, positive definite) and a Hermitian H
        N, n = case["N"], case["batch"]
        K = rng.standard_normal((n, N, N)) + 1j * rng.standard_normal((n, N, N))
        S = np.eye(N) + (K + K.conj().transpose(0, 2, 1)) * (0.2 / math.sqrt(N))
        H = rng.standard_normal((n, N, N)) + 1j * rng.standard_normal((n, N, N))
        return S, H + H.conj().transpose(0, 2, 1)
    if case["kind"] == "elements":
        R = np.sort(rng.uniform(-20.0, 20.0, case["positions"]))
        return float(rng.uniform(case["b_lo"], case["b_hi"])), case["v"] * (1.0 + 0.03 * rng.uniform(-1.0, 1.0)), R
    return _paths(case, rng) + (rng,)


def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda", 0)
    if kind == "solve":
        S, H = (w.colmajor(torch.from_numpy(x)).to(dev) for x in _inputs(case, seed))
        return dict(kind=kind, S0=S, H0=H, S=S.clone(), H=H.clone())
    if kind == "batch":
        sets, c0 = [], []
        for k, v in enumerate(float(s) for s in case["speeds"].split(",")):
            sc = _scan_case(case, v)
            g = w.Basis(_basis(sc))
            g.set_solve_mode(SOLVES[sc["solve"]])
            b, vv, zg, rng = _inputs(sc, 1000003 * (k + 1) + seed)
            sets.append((g, b, vv, zg))
            c0.append(torch.from_numpy(_amplitudes(sc, rng, b.size, g.N)).to(dev))
        c = [t.clone() for t in c0]
        return dict(kind=kind, c0=c0, c=c, bases=[s[0] for s in sets],
                    batch=w.Batch(sets, c, precision_mode=case["mode"]))
    basis = _basis(case)
    g = w.Basis(basis)
    if kind == "elements":
        b, v, z = _inputs(case, seed)
        S, H = (torch.zeros((z.size, g.N, g.N), dtype=torch.complex128, device=dev) for _ in range(2))
        return dict(kind=kind, g=g, b=b, v=v, z=z, S=S, H=H, mode=case["mode"])
    b, v, zg, rng = _inputs(case, seed)
    c0 = torch.from_numpy(_amplitudes(case, rng, b.size, g.N)).to(dev)
    state = dict(kind=kind, g=g, b=b, v=v, zg=zg, c0=c0, c=c0.clone())
    if kind == "gradient":
        return dict(state, weights=wi.observable_weights(basis), checkpoint=case["checkpoint"])
    g.set_solve_mode(SOLVES[case["solve"]])
    g.set_refine_iters(case["iters"])
    return dict(state, mode=case["mode"])


def run(state):
    kind = state["kind"]
    if kind == "elements":
        if state["mode"] == 0:
            S, H = state["g"].matrix_elements(state["b"], state["v"], state["z"], state["S"], state["H"])
        else:
            S, H = state["g"].matrix_elements_precision(state["b"], state["v"], state["z"], state["mode"], state["S"],
                                                        state["H"])
        return dict(S=S, H=H)
    if kind == "solve":
        state["S"].copy_(state["S0"])
        state["H"].copy_(state["H0"])
        w.solve(state["S"], state["H"])
        return dict(X=state["H"])
    if kind == "batch":
        for c, c0 in zip(state["c"], state["c0"]):
            c.copy_(c0)
        state["batch"].launch()
        state["batch"].status()
        return dict(c=state["c"], P=[w.probabilities(c) for c in state["c"]])
    c = state["c"]
    c.copy_(state["c0"])
    if kind == "gradient":
        c, P, grad = state["g"].propagate_adjoint(state["b"], state["v"], state["zg"], state["weights"],
                                                  state["checkpoint"], c=c)
        return dict(c=c, P=P, grad=grad)
    state["g"].propagate(state["b"], state["v"], state["zg"], c=c, precision_mode=state["mode"])
    return dict(c=c, P=w.probabilities(c))


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------


def _half(nmax, lmax, nbins):
    """Projectile states with q >= 0 in the molecular frame: the others follow by reflection."""
    return sum((l + 1) * (max(0, nmax - l) + nbins) for l in range(lmax + 1))


def _sizes(case):
    """(N_T, N_P, q >= 0 projectile states, nodes, radial functions of both centres)"""
    if case["kind"] == "gradient":
        NT, NP = _states(case["nmax"], case["lmax"], case["nbins"]) - 1, _states(case["nmax"], case["lmax"], case["nbins"])
        return NT, NP, _half(case["nmax"], case["lmax"], case["nbins"]), case["Geta"] * case["Gtau"]
    NT = _states(case["nmax"], case["lmax"], case["nbins"])
    if case["centres"] == 1:
        return NT, 0, 0, 0
    P = (case["nmax_P"], case["lmax_P"], case["nbins_P"])
    return NT, _states(*P), _half(*P), case["Geta"] * case["Gtau"]


def _propagate_flops(case, positions, path_steps):
    """Overlap and transfer sums over the nodes (two complex results from real tables), the direct blocks, the
    factorisation of S per position, and per RK4 stage H y and one solve."""
    NT, NP, half, G = _sizes(case)
    N = NT + NP
    lam = case["lmax"] + 1
    f = positions * (8.0 * NT * half * G + 2.0 * lam * (NT * NT + NP * NP))
    if NP:
        f += positions * (4.0 * NP * NP * NT + 4.0 / 3.0 * NP ** 3)
    return f + path_steps * 4.0 * (8.0 * N * N + 16.0 * NT * NP + 8.0 * NP * NP)


def work(case):
    kind = case["kind"]
    if kind == "solve":
        N, n = case["N"], case["batch"]
        return dict(bytes=3.0 * 16 * N * N * n, flops=n * (8.0 / 3.0 + 8.0) * N ** 3)
    if kind == "batch":
        parts = [work(_scan_case(case, float(s))) for s in case["speeds"].split(",")]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    NT, NP, half, G = _sizes(case)
    N = NT + NP
    if kind == "elements":
        n = case["positions"]
        return dict(bytes=2.0 * 16 * N * N * n,
                    flops=n * (8.0 * NT * half * G + 2.0 * (case["lmax"] + 1) * (NT * NT + NP * NP)))
    n, steps = case["paths"], case["steps"] * (0.75 if case.get("ragged") else 1.0)
    flops = _propagate_flops(case, n * (2 * steps + 1), n * steps)
    out = 3.0 * 16 * n * N
    return dict(bytes=out, flops=3.0 * flops if kind == "gradient" else flops)


# ---------------------------------------------------------------------------
# the method in plain numpy
# ---------------------------------------------------------------------------


def _clebsch(j1, m1, j2, m2, J, M):
    """<j1 m1 j2 m2 | J M> by Racah's sum."""
    f = math.factorial
    if m1 + m2 != M or abs(m1) > j1 or abs(m2) > j2 or abs(M) > J or not abs(j1 - j2) <= J <= j1 + j2:
        return 0.0
    pre = (2 * J + 1) * f(J + j1 - j2) * f(J - j1 + j2) * f(j1 + j2 - J) / f(j1 + j2 + J + 1)
    pre *= f(J + M) * f(J - M) * f(j1 - m1) * f(j1 + m1) * f(j2 - m2) * f(j2 + m2)
    s = 0.0
    for k in range(j1 + j2 - J + 1):
        d = (k, j1 + j2 - J - k, j1 - m1 - k, j2 + m2 - k, J - j2 + m1 + k, J - j1 - m2 + k)
        if min(d) >= 0:
            s += (-1) ** k / math.prod(f(x) for x in d)
    return s * math.sqrt(pre)


def _small_d(j, mp, m, beta):
    """Wigner d^j_{m' m}(beta), explicit sum."""
    f = math.factorial
    c, s = math.cos(beta / 2.0), math.sin(beta / 2.0)
    pre = math.sqrt(f(j + mp) * f(j - mp) * f(j + m) * f(j - m))
    t = 0.0
    for k in range(2 * j + 1):
        d = (j + m - k, k, mp - m + k, j - mp - k)
        if min(d) >= 0:
            t += (-1) ** (mp - m + k) * c ** (2 * j + m - mp - 2 * k) * s ** (mp - m + 2 * k) / math.prod(f(x) for x in d)
    return t * pre


def _legendre(lmax, x):
    """{(l, m): P_l^m(x)} for 0 <= m <= l <= lmax with the Condon-Shortley phase."""
    p = {}
    s = np.sqrt((1.0 - x) * (1.0 + x))
    for m in range(lmax + 1):
        p[m, m] = (-1.0) ** m * math.prod(range(1, 2 * m, 2)) * s ** m
        if m < lmax:
            p[m + 1, m] = (2 * m + 1) * x * p[m, m]
        for l in range(m + 2, lmax + 1):
            p[l, m] = ((2 * l - 1) * x * p[l - 1, m] - (l + m - 1) * p[l - 2, m]) / (l - m)
    return p


def _bessel(dmax, x):
    """J_0(x) .. J_dmax(x) as Fourier coefficients of exp(i x sin t): the trapezoid rule on the circle, exact up to
    aliasing from orders far above the argument."""
    out = np.zeros((dmax + 1, x.size))
    size = np.maximum(64, 2 ** np.ceil(np.log2(1.3 * x + 2 * dmax + 48))).astype(int)
    for n in np.unique(size):
        at = np.nonzero(size == n)[0]
        for part in np.array_split(at, max(1, at.size * int(n) // 4000000)):
            t = np.exp(1j * np.outer(x[part], np.sin(2.0 * np.pi * np.arange(n) / n)))
            out[:, part] = (np.fft.fft(t, axis=1)[:, :dmax + 1].real / n).T
    return out


def _stencil(r, x):
    """Nodes and weights of the 5-point Lagrange interpolation at x."""
    s = np.clip(np.searchsorted(r, x, side="right") - 3, 0, r.size - 5)
    nodes = s[..., None] + np.arange(5)
    rn = r[nodes]
    L = np.ones(rn.shape)
    for a in range(5):
        for b in range(5):
            if a != b:
                L[..., a] *= (x - rn[..., b]) / (rn[..., a] - rn[..., b])
    return nodes, L


def _direct_tables(grid, c):
    """Eq. 7 table F[a, b, lam][R on the grid] (by radial pair and multipole) and Eq. 6's angular factors."""
    key = "_cases_direct"
    if hasattr(c, key):
        return getattr(c, key)
    r, wt = grid.r, grid.w
    lmax, n = int(c.rad_l.max()), c.n_rad
    F = {}
    for lam in range(2 * lmax + 1):
        ok = [(a, b) for a in range(n) for b in range(a, n) if abs(int(c.rad_l[a]) - int(c.rad_l[b])) <= lam
              <= int(c.rad_l[a]) + int(c.rad_l[b]) and (int(c.rad_l[a]) + int(c.rad_l[b]) + lam) % 2 == 0]
        if ok:
            a, b = np.array(ok).T
            g = c.f[a] * c.f[b] * (wt * r * r)
            inner = np.cumsum(g * r ** lam, axis=1)
            outer = g / r ** (lam + 1)
            outer = np.cumsum(outer[:, ::-1], axis=1)[:, ::-1] - outer
            F[lam] = a, b, inner / r ** (lam + 1) + outer * r ** lam
    ang = np.zeros((2 * lmax + 1, c.N, c.N))
    memo = {}
    for i in range(c.N):
        for j in range(c.N):
            lp, mp, l, m = int(c.st_l[i]), int(c.st_m[i]), int(c.st_l[j]), int(c.st_m[j])
            if (lp, mp, l, m) not in memo:
                v = np.zeros(2 * lmax + 1)
                for lam in range(abs(lp - l), lp + l + 1, 2):
                    mu = mp - m
                    if abs(mu) <= lam:
                        q = math.sqrt((2 * l + 1) / (2 * lp + 1) * math.factorial(lam - abs(mu)) / math.factorial(lam + abs(mu)))
                        sign = (-1.0) ** mu if mu < 0 else 1.0
                        v[lam] = q * sign * _clebsch(lam, 0, l, 0, lp, 0) * _clebsch(lam, mu, l, m, lp, mp)
                memo[lp, mp, l, m] = v
            ang[:, i, j] = memo[lp, mp, l, m]
    setattr(c, key, (F, ang))
    return F, ang


def _direct(grid, c, charge, R, cth, parity):
    """Eq. 6 block without its energy phases, at every R: [positions, N, N]."""
    F, ang = _direct_tables(grid, c)
    r, n = grid.r, c.n_rad
    inside = R <= r[-1]
    nodes, L = _stencil(r, np.where(inside, R, r[-1]))
    P = _legendre(int(2 * c.rad_l.max()), cth)
    dm = np.abs(c.st_m[:, None] - c.st_m[None, :])
    D = np.zeros((R.size, c.N, c.N))
    for lam, (a, b, tab) in F.items():
        at = np.einsum("apk,pk->pa", tab[:, nodes], L)
        at = np.where(inside[:, None], at, tab[None, :, -1] * ((r[-1] / R) ** (lam + 1))[:, None])
        full = np.zeros((R.size, n, n))
        full[:, a, b] = at
        full[:, b, a] = at
        Pm = np.stack([P[lam, m] if m <= lam else np.zeros(R.size) for m in range(int(dm.max()) + 1)], axis=1)
        D += (-charge * parity ** lam) * ang[lam] * Pm[:, dm] * full[:, c.st_rad[:, None], c.st_rad[None, :]]
    return D


def _theta_states(c, x):
    """Theta_{l q}(x) of every state, m read as the molecular-frame q."""
    P = _legendre(int(c.rad_l.max()), x)
    f = math.factorial
    rows = []
    for l, m in zip(c.st_l.tolist(), c.st_m.tolist()):
        q = abs(m)
        rows.append(math.sqrt((2 * l + 1) / 2.0 * f(l - q) / f(l + q)) * ((-1.0) ** q if m < 0 else 1.0) * P[l, q])
    return np.array(rows)


def _rotation(c, theta):
    D = np.zeros((c.N, c.N))
    first = 0
    while first < c.N:
        l = int(c.st_l[first])
        k = 2 * l + 1
        if first and int(c.st_l[first - 1]) == l:
            D[first:first + k, first:first + k] = D[first - k:first, first - k:first]
        else:
            D[first:first + k, first:first + k] = [[_small_d(l, mp, m, theta) for m in range(-l, l + 1)]
                                                   for mp in range(-l, l + 1)]
        first += k
    return D


def _two_centre(basis, b, v, z):
    """K and Q of Eq. 9 and Eq. 8 at one position, without the energy phases."""
    T, P, q, r = basis.T, basis.P, basis.quad, basis.grid.r
    R = math.sqrt(b * b + z * z)
    eta, tau = np.meshgrid(1.0 + q.s / (q.gamma * R), q.tau, indexing="ij")
    wt = np.outer(q.ws / (q.gamma * R), q.wtau).ravel()
    eta, tau = eta.ravel(), tau.ravel()
    # nodes beyond the radial grid of either centre contribute nothing
    keep = (0.5 * R * (eta + tau) <= r[-1]) & (0.5 * R * (eta - tau) <= r[-1])
    eta, tau, wt = eta[keep], tau[keep], wt[keep]
    rT, rP = 0.5 * R * (eta + tau), 0.5 * R * (eta - tau)
    A = []
    for c, rad, cos in ((T, rT, (eta * tau + 1.0) / (eta + tau)), (P, rP, (eta * tau - 1.0) / (eta - tau))):
        nodes, L = _stencil(r, rad)
        f = np.einsum("agk,gk->ag", c.f[:, nodes], L)
        A.append(f[c.st_rad] * _theta_states(c, cos))
    base = R ** 3 / 8.0 * wt * (eta * eta - tau * tau) * np.exp(0.5j * v * z * eta * tau)
    dmax = int(T.st_l.max() + P.st_l.max())
    J = _bessel(dmax, 0.5 * v * b * np.sqrt((eta * eta - 1.0) * (1.0 - tau * tau)))
    W = {}
    for d in range(dmax + 1):
        W[d] = base * (-1j) ** d * J[d]
    out = []
    for u in (1.0, -basis.Z_T / rT):
        X = np.zeros((T.N, P.N), dtype=np.complex128)
        for qp in np.unique(T.st_m):
            rows = np.nonzero(T.st_m == qp)[0]
            for qq in np.unique(P.st_m):
                cols = np.nonzero(P.st_m == qq)[0]
                Wd = W[abs(int(qq) - int(qp))] * u
                # (-i)^d J_d is even in d
                X[np.ix_(rows, cols)] = (A[0][rows] * Wd.real) @ A[1][cols].T + 1j * ((A[0][rows] * Wd.imag) @ A[1][cols].T)
        th = math.acos(z / R)
        out.append(_rotation(T, th) @ X @ _rotation(P, th).T)
    return out


def _elements(basis, b, v, z):
    """S and H at the positions z of the path (b, v): [positions, N, N] each."""
    T, P = basis.T, basis.P
    z = np.asarray(z, dtype=np.float64)
    R = np.sqrt(b * b + z * z)
    eps = T.st_eps if P is None else np.concatenate([T.st_eps, P.st_eps])
    ph = np.exp(1j * eps[None, :] * z[:, None] / v)
    ph = ph[:, :, None] * ph.conj()[:, None, :]
    NT, N = T.N, basis.N
    S = np.zeros((z.size, N, N), dtype=np.complex128)
    S[:, range(N), range(N)] = 1.0
    H = np.zeros((z.size, N, N), dtype=np.complex128)
    H[:, :NT, :NT] = _direct(basis.grid, T, basis.Z_P, R, z / R, 1.0)
    if P is not None:
        H[:, NT:, NT:] = _direct(basis.grid, P, basis.Z_T, R, z / R, -1.0)
        for k, zk in enumerate(z.tolist()):
            K, Q = _two_centre(basis, b, v, zk)
            S[k, :NT, NT:], H[k, :NT, NT:] = K, Q
            S[k, NT:, :NT], H[k, NT:, :NT] = K.conj().T, Q.conj().T
        S *= ph
    return S, H * ph


def _rk4(basis, b, v, z, c):
    """Algorithm 1 along one path, in blocks of positions."""
    def slopes(at):
        S, H = _elements(basis, b, v, at)
        return (-1j / v) * (H if basis.P is None else np.linalg.solve(S, H))

    last = None
    for s in range(0, z.size - 1, 32):
        zz = z[s:s + 33]
        at = np.empty(2 * zz.size - 1)
        at[::2], at[1::2] = zz, (zz[:-1] + zz[1:]) / 2.0
        M = slopes(at if last is None else at[1:])
        M = M if last is None else np.concatenate([last, M])
        for k, h in enumerate(np.diff(zz).tolist()):
            k1 = M[2 * k] @ c
            k2 = M[2 * k + 1] @ (c + 0.5 * h * k1)
            k3 = M[2 * k + 1] @ (c + 0.5 * h * k2)
            k4 = M[2 * k + 2] @ (c + h * k3)
            c = c + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        last = M[-1:]
    return c


def exact(case, seed):
    """What ``run`` returns, in FP64 numpy; None where that would take too long (and for the gradient)."""
    kind = case["kind"]
    if kind in ("batch", "gradient"):
        return None
    if kind == "solve":
        S, H = _inputs(case, seed)
        return dict(X=np.ascontiguousarray(np.linalg.solve(S, H).transpose(0, 2, 1)))
    NT, NP, half, G = _sizes(case)
    per = 2e-3 * (NT / 59.0) ** 2 if NP == 0 else 0.03 + NT * NP * G * 16 / 2e10 + 2e-10 * (NT + NP) ** 3
    count = case["positions"] if kind == "elements" else case["paths"] * 2 * case["steps"]
    if count * per > 18.0 and not (NP == 0 and NT < 80):
        return None
    basis = _basis(case)
    if kind == "elements":
        S, H = _elements(basis, *_inputs(case, seed))
        return {k: np.ascontiguousarray(x.transpose(0, 2, 1)) for k, x in (("S", S), ("H", H))}
    b, v, zg, rng = _inputs(case, seed)
    c0 = _amplitudes(case, rng, b.size, basis.N)
    c = np.stack([_rk4(basis, float(b[p]), v, zg[p], c0[p]) for p in range(b.size)])
    return dict(c=c, P=np.abs(c) ** 2)
