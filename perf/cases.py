"""Performance cases of the trajectory framework: the calls its users make, over the sizes they make them at.

Each case names a call of the public binding (paper_2312_02322_gb300.api), its system and its
trajectories.  The systems are the repository's own seeded workloads (diatom + atom, asymmetric top + atom,
asymmetric top + linear rotor, the log-grid truncated setup, the rate set); trajectories (energies, impact
parameters, initial states) come from the seed.

Trajectories of the FP64 paths run to the stop rule (R >= r_end moving outwards).  Those of the
mixed-precision paths are followed for a fixed time (a multiple of the flight time 2 r0 / v of their
energy, or a step cap), as for time-resolved populations: their step counts are given, not decided by
the last bits of an FP32 sum.

Populations and amplitudes of the mixed paths are FP32 numbers that the library stores in FP64 arrays; they
are returned as the FP32 numbers they are (the conversion loses nothing).
"""
import math

import numpy as np
import torch

from paper_2312_02322_gb300 import api
from paper_2312_02322_gb300 import inputs as W

SIGMA_GROUPS = 4


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # a first look at a small system: plain FP64 path, host arrays in and out, amplitudes too
        # (N = 49, 32 impact parameters, E = 500 cm^-1: the smallest workload of the repository)
        dict(name="fp64_n49_host", kind="traj", rotor="diatom", jmax=6, path="plain", precision="fp64", n=32,
             e_lo=500.0, e_hi=500.0, b_max=12.0, r0=30.0, follow=0.0, cap=1000000, host=True, sigma=True, tol=0.0),
        # a cross-section set in FP64 (N = 441, device arrays, then the cross sections)
        dict(name="fp64_n441_plain", kind="traj", rotor="diatom", jmax=20, path="plain", precision="fp64", n=256,
             e_lo=1000.0, e_hi=3000.0, b_max=10.0, r0=12.0, follow=0.0, cap=1000000, host=False, sigma=True, tol=0.0),
        # molecule + molecule (asymmetric top + linear rotor, N = 210, nine terms), FP64, factorised coupling
        dict(name="fp64_molmol", kind="traj", rotor="molmol", jmax=2, path="factorised", precision="fp64", n=304,
             e_lo=300.0, e_hi=1500.0, b_max=8.0, r0=10.0, follow=0.0, cap=1000000, host=False, sigma=True, tol=0.0),
        # a handful of trajectories for a short time in mixed precision from host arrays: the cost of a call
        dict(name="fp32_few_host", kind="traj", rotor="diatom", jmax=10, path="factorised", precision="fp32", n=8,
             e_lo=500.0, e_hi=2000.0, b_max=6.0, r0=8.0, follow=0.8, cap=256, host=True, sigma=False, tol=0.0),
        # the headline workload: N = 441, 3072 trajectories of uneven length in mixed precision
        dict(name="fp32_n441", kind="traj", rotor="diatom", jmax=20, path="factorised", precision="fp32", n=3072,
             e_lo=100.0, e_hi=3000.0, b_max=15.0, r0=20.0, follow=0.8, cap=1000000, host=False, sigma=False, tol=0.0),
        # the larger basis of the same comparison, N = 1600
        dict(name="fp32_n1600", kind="traj", rotor="diatom", jmax=39, path="factorised", precision="fp32", n=512,
             e_lo=1000.0, e_hi=3000.0, b_max=12.0, r0=15.0, follow=0.8, cap=1000000, host=False, sigma=False, tol=0.0),
        # the serving mix: four bases (N = 49, 121, 441, 1600 in 1:2:4:1) in one call
        dict(name="fp32_mix", kind="mix", n=2048, e_lo=10.0, e_hi=5000.0, b_max=15.0, r0=20.0, follow=0.8, cap=6000),
        # asymmetric top + atom, N = 1580, 28 terms: the tensor-core path
        dict(name="bf16x3_asym1580", kind="traj", rotor="asym", jmax=12, path="factorised", precision="bf16x3",
             n=1024, e_lo=100.0, e_hi=2000.0, b_max=10.0, r0=12.0, follow=0.8, cap=160, host=False, sigma=False,
             tol=0.0),
        # the paper-scale setup (log grid, |M| truncation, N = 40401), sparse FP32 path
        dict(name="sparse_n40401", kind="sparse", jmax=200, lam_max=12, n=512, e_lo=400.0, e_hi=5000.0, b_max=5.0,
             r0=8.0, cap=48),
        # gradients of the cross sections with respect to the ten PES parameters: FP64 and mixed adjoint
        dict(name="adjoint_fp64_n441", kind="adjoint", jmax=20, precision="fp64", n=128, e_lo=1000.0, e_hi=3000.0,
             b_max=6.0, r0=8.0, ckpt=64),
        dict(name="adjoint_fp32_n441", kind="adjoint", jmax=20, precision="fp32", n=256, e_lo=1000.0, e_hi=3000.0,
             b_max=6.0, r0=8.0, ckpt=64),
        # rate coefficients of the paper's 1032 channels at ten energies and five temperatures
        dict(name="rates_1032", kind="rates", levels=1032, temps=5, t_lo=10.0, t_hi=1000.0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, at most as costly as the largest listed one."""
    kind = rng.choice(["fp64", "fp64", "molmol", "fp32", "fp32", "mix", "bf16x3", "sparse", "adjoint", "rates"])
    e_lo = round(rng.uniform(200.0, 1500.0), 1)
    e_hi = round(e_lo * rng.uniform(1.0, 3.0), 1)
    r0 = round(rng.uniform(8.0, 12.0), 2)
    b_max = round(rng.uniform(3.0, 0.75 * r0), 2)
    if kind == "fp64":
        jmax = rng.choice([2, 3, 6, 9, 13, 20, 23])
        most = max(1, int(4e8 / ((jmax + 1) ** 2 * 4000)))  # states x steps of the N = 441 case
        return dict(kind="traj", rotor="diatom", jmax=jmax, path=rng.choice(["plain", "factorised"]),
                    precision="fp64", n=_logint(rng, 1, min(1024, most)), e_lo=e_lo + 300.0, e_hi=e_hi + 300.0,
                    b_max=b_max, r0=r0, follow=0.0, cap=1000000, host=rng.random() < 0.5, sigma=True,
                    tol=rng.choice([0.0, 0.0, 1e-6]))
    if kind == "molmol":
        return dict(kind="traj", rotor="molmol", jmax=rng.choice([1, 2]), path=rng.choice(["plain", "factorised"]),
                    precision="fp64", n=_logint(rng, 8, 400), e_lo=e_lo + 300.0, e_hi=e_hi + 300.0,
                    b_max=b_max, r0=r0, follow=0.0, cap=1000000, host=rng.random() < 0.5, sigma=True, tol=0.0)
    if kind == "fp32":
        jmax = rng.randint(3, 39)
        n = _logint(rng, 1, 3072)
        cap = max(16, min(_logint(rng, 32, 8000), int(1.2e10 / (n * (jmax + 1) ** 2))))
        return dict(kind="traj", rotor="diatom", jmax=jmax, path="factorised", precision="fp32", n=n, e_lo=e_lo,
                    e_hi=e_hi, b_max=b_max, r0=r0, follow=0.8, cap=cap, host=rng.random() < 0.3, sigma=False, tol=0.0)
    if kind == "mix":
        return dict(kind="mix", n=_logint(rng, 64, 2048), e_lo=20.0, e_hi=e_hi + 1000.0, b_max=b_max, r0=r0,
                    follow=0.8, cap=_logint(rng, 200, 4000))
    if kind == "bf16x3":
        jmax = rng.randint(5, 12)
        return dict(kind="traj", rotor="asym", jmax=jmax, path="factorised", precision="bf16x3",
                    n=_logint(rng, 16, 1024), e_lo=e_lo, e_hi=e_hi, b_max=b_max, r0=r0, follow=0.8,
                    cap=rng.randint(24, 160), host=rng.random() < 0.3, sigma=False, tol=0.0)
    if kind == "sparse":
        return dict(kind="sparse", jmax=_logint(rng, 40, 160), lam_max=rng.choice([6, 8, 12]), n=_logint(rng, 16, 700),
                    e_lo=e_lo, e_hi=e_hi, b_max=round(min(b_max, 6.0), 2), r0=r0, cap=rng.randint(12, 48))
    if kind == "adjoint":
        return dict(kind="adjoint", jmax=rng.choice([5, 9, 13, 20]), precision=rng.choice(["fp64", "fp32"]),
                    n=_logint(rng, 4, 152), e_lo=e_lo + 800.0, e_hi=e_hi + 800.0, b_max=round(min(b_max, 6.0), 2), r0=8.0,
                    ckpt=rng.choice([16, 50, 64]))
    return dict(kind="rates", levels=_logint(rng, 30, 1032), temps=rng.randint(1, 8), t_lo=10.0,
                t_hi=round(rng.uniform(300.0, 2000.0), 1))


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _params(case):
    if case["kind"] == "sparse":
        return W.sparse_pes_params(jmax=case["jmax"], lam_max=case["lam_max"])
    rotor = case.get("rotor", "diatom")
    if rotor == "molmol":
        return W.molmol_params(j1max=case["jmax"])
    if rotor == "asym":
        return W.asym_pes_params(jmax=case["jmax"])
    return W.diatom_pes_params(jmax=case["jmax"], n_grid=400 if case["jmax"] > 6 else 200)


def _trunc():
    return (float(W.cm(W.PAPER_TRUNC_CM)), *W.PAPER_TRUNC_R)


def _system(case, p):
    if case["kind"] == "sparse":
        return api.System.diatom(p, path="plain", precision="fp32", grid="log", trunc=_trunc())
    if case["kind"] == "adjoint":
        return api.System.diatom(p, path="factorised", precision=case["precision"], with_params=True)
    if case["rotor"] == "molmol":
        return api.System.molmol(p, path=case["path"], precision=case["precision"])
    if case["rotor"] == "asym":
        return api.System.asym_top(p, path=case["path"], precision=case["precision"])
    return api.System.diatom(p, path=case["path"], precision=case["precision"],
                             adapt=(case["tol"], 16) if case.get("tol") else None)


def _steps(case, e, mu, r0, dt):
    """Step caps: the fixed time follow * 2 r0 / v of each energy, at most cap; the cap alone otherwise."""
    if not case.get("follow"):
        return np.full(len(e), case.get("cap", 1000000), np.int32)
    t = case["follow"] * 2.0 * r0 * np.sqrt(mu / (2.0 * e))
    return np.minimum(np.ceil(t / dt), case["cap"]).astype(np.int32)


def _trajs(case, seed, mus, init_of, system=None):
    """mqct_traj array: E log-uniform on [e_lo, e_hi], b uniform on [0, b_max]; init_of(rng, i) is a state."""
    rng = np.random.default_rng(seed)
    n, dt, r0 = case["n"], 5.0, case["r0"]
    tr = np.zeros(n, api.TRAJ_DTYPE)
    e = np.asarray(W.cm(np.exp(rng.uniform(math.log(case["e_lo"]), math.log(case["e_hi"] + 1e-9), n))))
    tr["e_coll"], tr["b"] = e, rng.uniform(0.0, case["b_max"], n)
    tr["r0"], tr["dt"] = r0, dt
    # a trajectory of given length never meets the stop rule
    fixed = bool(case.get("follow")) or case["kind"] == "sparse"
    tr["r_end"] = 4.0 * r0 if fixed else r0
    s = np.zeros(n, np.int32) if system is None else system
    tr["system_idx"] = s
    mu = np.asarray(mus)[s]
    tr["max_steps"] = _steps(case, e, mu, r0, dt)
    tr["init_state"] = [init_of(rng, i) for i in range(n)]
    return tr


def _low_state(sys_):
    def f(rng, i):
        j = int(rng.integers(0, 3))
        j = min(j, int(sys_.j.max()))
        return sys_.state(j, int(rng.integers(-j, j + 1)))
    return f


def _to_device(tr):
    return torch.from_numpy(tr.view(np.uint8).copy()).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "rates":
        temps = np.geomspace(case["t_lo"], case["t_hi"], case["temps"])
        rs = W.rate_set(n_levels=case["levels"], temps_k=tuple(temps), seed=seed)
        return dict(case=case, rs=rs, sigma=torch.from_numpy(rs.sigma).cuda())
    if kind == "mix":
        jmaxes, share = [6, 10, 20, 39], [1, 2, 4, 1]
        systems = [api.System.diatom(W.diatom_pes_params(jmax=j, n_grid=400), path="factorised", precision="fp32")
                   for j in jmaxes]
        rng = np.random.default_rng(seed + 77)
        # shares of the bases fixed, their order in the call random
        sidx = rng.permutation(np.searchsorted(np.cumsum(share) / 8.0, np.arange(case["n"]) / case["n"],
                                               side="right")).astype(np.int32)
        tr = _trajs(case, seed, [s.mu for s in systems], lambda r, i: systems[sidx[i]].state(0, 0), sidx)
        rows = [torch.from_numpy(np.nonzero(sidx == i)[0]).cuda() for i in range(4)]
        return dict(case=case, systems=systems, trajs=_to_device(tr), rows=rows)
    p = _params(case)
    sys_ = _system(case, p)
    # diatom and molecule-molecule runs start in the lowest levels, the asymmetric top in its ground level
    low = _low_state(sys_) if isinstance(p, W.DiatomParams) else (lambda r, i: 0)
    tr = _trajs(case, seed, [sys_.mu], low)
    rng = np.random.default_rng(seed + 5)
    group = rng.integers(0, SIGMA_GROUPS, case["n"]).astype(np.int32)
    weight = 2.0 * np.pi * case["b_max"] * tr["b"] / case["n"]
    st = dict(case=case, p=p, sys=sys_, tr=tr, weight=weight, group=group)
    if kind == "adjoint":
        st["dL"] = rng.normal(size=(SIGMA_GROUPS, sys_.n_levels))
    if kind == "sparse" or not case.get("host", True):
        st["trajs"] = _to_device(tr)
        st["weight_d"], st["group_d"] = torch.from_numpy(weight).cuda(), torch.from_numpy(group).cuda()
    return st


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def _ints(diag):
    """steps and status of the diagnostics of a device call"""
    return diag.view(-1, api.DIAG_DTYPE.itemsize)[:, :8].contiguous().view(torch.int32)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "rates":
        rs = st["rs"]
        sym, rate = api.rate_coefficients(st["sigma"], rs.u, rs.energy, rs.g, rs.mu, rs.kT)
        return {"sigma_sym": sym, "rate": rate}
    if kind == "mix":
        pop, _, diag = api.propagate(st["systems"], st["trajs"], device=True)
        return {"pop": [pop[r, :s.n].float() for r, s in zip(st["rows"], st["systems"])], "ints": _ints(diag)}
    if kind == "adjoint":
        return api.adjoint(st["sys"], st["tr"], st["weight"], st["group"], SIGMA_GROUPS, st["dL"], case["ckpt"])
    fp64 = case.get("precision") == "fp64"
    if kind == "traj" and case["host"]:
        pop, amp, diag = api.propagate(st["sys"], st["tr"], want_amp=True, device=False)
        if not fp64:
            return {"pop": pop.astype(np.float32), "amp": amp.astype(np.complex64),
                    "steps": diag["steps"], "status": diag["status"]}
        sig = api.cross_sections(st["sys"], pop, st["weight"], st["group"], SIGMA_GROUPS)
        return {"pop": pop, "amp": amp, "steps": diag["steps"], "status": diag["status"], "sigma": sig}
    pop, _, diag = api.propagate(st["sys"], st["trajs"], device=True)
    if not fp64:
        return {"pop": pop.float(), "ints": _ints(diag)}
    sig = api.cross_sections(st["sys"], pop, st["weight_d"], st["group_d"], SIGMA_GROUPS)
    return {"pop": pop, "ints": _ints(diag), "sigma": sig}


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
def _band(jmax, lam):
    """non-zeros of G^lambda of a linear rotor (|dj| <= lambda, dj = lambda mod 2)"""
    return sum(sum(1 for d in range(-lam, lam + 1, 2) if abs(m) <= j + d <= jmax and (m or d + lam >= 0))
               for j in range(jmax + 1) for m in range(-j, j + 1))


def _mean_steps(case, mu):
    e = float(W.cm(math.sqrt(case["e_lo"] * case["e_hi"])))
    v = math.sqrt(2.0 * e / mu)
    if case["kind"] == "sparse":
        return float(case["cap"])
    full = 2.0 * case["r0"] / (v * 5.0)
    if case.get("follow"):
        return min(case["follow"] * full, case["cap"])
    return 0.75 * full / (8.0 if case.get("tol") else 1.0)  # turning point and impact parameter; larger steps


def work(case):
    kind = case["kind"]
    if kind == "rates":
        L, T, K = case["levels"], case["temps"], 10
        return {"bytes": 8.0 * L * L * (2 * K + T), "flops": 0.5 * L * L * (2.0 * K * K + T * (10.0 * K + 60.0))}
    mu = 1.8 * W.AMU_ME if kind == "sparse" or case.get("rotor") == "molmol" else (
        3.3 * W.AMU_ME if case.get("rotor") == "asym" else 4.0 * W.AMU_ME)
    steps, n = _mean_steps(case, mu), case["n"]
    if kind == "mix":
        parts = [(6, 1 / 8), (10, 2 / 8), (20, 4 / 8), (39, 1 / 8)]
        flops = byts = 0.0
        for jmax, f in parts:
            N = (jmax + 1) ** 2
            flops += f * n * steps * 4 * (4.0 * sum(_band(jmax, l) for l in range(1, 5)) + 80.0 * N)
            byts += f * n * (56 + 8 + 4 * N)
        return {"bytes": byts, "flops": flops}
    if kind == "sparse":
        N = (case["jmax"] + 1) ** 2
        nnz = 12.0 * N
        return {"bytes": n * (64.0 + 8.0 * N) + 16.0 * nnz, "flops": n * steps * 4 * (10.0 * nnz + 60.0 * N)}
    if case.get("rotor") == "molmol":
        N, L = (210, 9) if case["jmax"] == 2 else (84, 9)
        nnz = 0.05 * N * N * L
    elif case.get("rotor") == "asym":
        N = min(1600, sum((2 * J + 1) ** 2 for J in range(case["jmax"] + 1)))
        L, nnz = 28, 28 * N * 15.0
    else:
        N, L = (case["jmax"] + 1) ** 2, 5
        nnz = sum(_band(case["jmax"], l) for l in range(1, 5))
    flops = n * steps * 4 * (4.0 * nnz + (8.0 * L + 40.0) * N)
    byts = n * (64.0 + 8.0 * N) + 12.0 * nnz + 32.0 * L * 400
    if kind == "adjoint":
        flops *= 4.0  # the forward pass and its reverse (about three forward passes)
        byts = n * 64.0 + 12.0 * nnz + 32.0 * (L + 10 * L) * 400
    return {"bytes": byts, "flops": flops}


# ------------------------------------------------------------------------------------------------
# the same results in plain FP64 torch and numpy (no code of the framework beyond its input numbers)
# ------------------------------------------------------------------------------------------------
def _legendre_G(jmax, lams):
    """<j+d m|P_lambda|j m> for every state s = j^2 + j + m and d = -lmax..lmax: [L][D][N] (Gauss-Legendre)"""
    lmax = max(lams)
    N, D = (jmax + 1) ** 2, 2 * lmax + 1
    x, w = np.polynomial.legendre.leggauss(jmax + lmax // 2 + 2)
    P = [np.ones_like(x), x.copy()]
    for l in range(1, lmax + 1):
        P.append(((2 * l + 1) * x * P[l] - l * P[l - 1]) / (l + 1))
    G = np.zeros((len(lams), D, N))
    pmm = np.full_like(x, math.sqrt(0.5))
    s2 = np.sqrt(1.0 - x * x)
    for m in range(jmax + 1):
        if m > 0:
            pmm = pmm * s2 * math.sqrt((2 * m + 1) / (2.0 * m))
        T = [pmm]
        if m < jmax:
            T.append(x * math.sqrt(2 * m + 3) * pmm)
        for j in range(m + 2, jmax + 1):
            a = math.sqrt((4.0 * j * j - 1) / (j * j - m * m))
            b = math.sqrt(((j - 1.0) ** 2 - m * m) / (4.0 * (j - 1.0) ** 2 - 1))
            T.append(a * (x * T[-1] - b * T[-2]))
        T = np.array(T[: jmax - m + 1])
        js = np.arange(m, jmax + 1)
        for li, lam in enumerate(lams):
            M = (T * (w * P[lam])) @ T.T
            for d in range(-lam, lam + 1):
                if (d + lam) % 2:
                    continue
                ok = (js + d >= m) & (js + d <= jmax)
                jj = js[ok]
                v = M[jj - m, jj + d - m]
                for mm in ({m, -m}):
                    G[li, d + lmax, jj * jj + jj + mm] = v
    return G, lmax


def _splines(p, log):
    """clamped cubic spline coefficients [L][n-1][4] of v_lambda in R (or ln R), first knot and spacing"""
    R = p.r_min * (p.r_max / p.r_min) ** (np.arange(p.n_grid) / (p.n_grid - 1)) if log else \
        p.r_min + np.arange(p.n_grid) * ((p.r_max - p.r_min) / (p.n_grid - 1))
    X0, X1 = (math.log(p.r_min), math.log(p.r_max)) if log else (p.r_min, p.r_max)
    h = (X1 - X0) / (p.n_grid - 1)
    out = []
    for l in range(p.n_terms):
        def f(r):
            e = p.A[l] * np.exp(-p.beta[l] * r)
            return e if l else e - p.c6 * r ** -6.0 * (1.0 - np.exp(-(r / p.rd) ** 6))

        def g(r):
            e = -p.beta[l] * p.A[l] * np.exp(-p.beta[l] * r)
            z = math.exp(-(r / p.rd) ** 6)
            return e if l else e + 6.0 * p.c6 * r ** -7.0 * (1.0 - z) - p.c6 * r ** -6.0 * z * 6.0 * r ** 5 / p.rd ** 6
        v = f(R)
        n = len(R)
        A, b = np.zeros((n, n)), np.zeros(n)
        A[0, 0] = A[-1, -1] = 1.0
        b[0] = g(p.r_min) * (p.r_min if log else 1.0)
        b[-1] = g(p.r_max) * (p.r_max if log else 1.0)
        i = np.arange(1, n - 1)
        A[i, i - 1], A[i, i], A[i, i + 1] = 1.0, 4.0, 1.0
        b[1:-1] = 3.0 * (v[2:] - v[:-2]) / h
        m = np.linalg.solve(A, b)
        dv = (v[1:] - v[:-1]) / h
        out.append(np.stack([v[:-1], m[:-1], (3 * dv - 2 * m[:-1] - m[1:]) / h, (m[:-1] + m[1:] - 2 * dv) / h ** 2], 1))
    return np.array(out), X0, h


def _exact_diatom(case, p, tr, log=False, trunc=None):
    """The RK4 map of Eqs. 4-10 on complex128 tensors, one column per trajectory."""
    dev = torch.device("cuda")
    lams = list(range(p.n_terms))
    G, lmax = _legendre_G(p.jmax, lams)
    D, N, B = 2 * lmax + 1, (p.jmax + 1) ** 2, len(tr)
    j = np.concatenate([np.full(2 * a + 1, a) for a in range(p.jmax + 1)])
    m = np.concatenate([np.arange(-a, a + 1) for a in range(p.jmax + 1)])
    idx = np.zeros((D, N), np.int64)
    for d in range(-lmax, lmax + 1):
        jj = j + d
        ok = (jj >= np.abs(m)) & (jj <= p.jmax)
        idx[d + lmax] = np.where(ok, jj * jj + jj + m, np.arange(N))
    coef, X0, h = _splines(p, log)

    def v_at(R):
        X = math.log(R) if log else R
        k = min(max(int(math.floor((X - X0) / h)), 0), p.n_grid - 2)
        x = X - (X0 + k * h)
        return coef[:, k] @ np.array([1.0, x, x * x, x ** 3])
    if trunc is not None:
        keep = np.zeros((D, N), bool)
        for R in trunc[1:]:
            keep |= np.abs(np.einsum("l,ldn->dn", v_at(R), G)) > trunc[0]
        G = G * keep
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    Gt = T(G.transpose(1, 2, 0)).reshape(D * N, -1)
    it, ct = T(idx), T(coef)
    au = T(np.sqrt(np.maximum(0, j * (j + 1) - m * (m + 1)))).unsqueeze(1)
    ad = T(np.sqrt(np.maximum(0, j * (j + 1) - m * (m - 1)))).unsqueeze(1)
    up, dn = T(np.where(m < j, np.arange(N) + 1, np.arange(N))), T(np.where(m > -j, np.arange(N) - 1, np.arange(N)))
    En = T(p.bconst * j * (j + 1.0)).unsqueeze(1)
    mu = p.mu
    e, b, dt = T(tr["e_coll"]), T(tr["b"]), float(tr["dt"][0])
    r0, rend = T(tr["r0"]), T(tr["r_end"])
    ms = T(tr["max_steps"].astype(np.int64))
    init = T(tr["init_state"].astype(np.int64))
    Gd = T(G[:, lmax])
    m00 = (T(v_at(case["r0"])).unsqueeze(1) * Gd[:, init]).sum(0)
    A = torch.zeros((N, B), dtype=torch.complex128, device=dev)
    A[init, torch.arange(B, device=dev)] = 1.0
    lz = b * torch.sqrt(2.0 * mu * e)
    q = torch.stack([r0, -torch.sqrt(2.0 * mu * (e - m00) - (lz / r0) ** 2), torch.zeros_like(e), lz])
    steps, done = torch.zeros(B, dtype=torch.int64, device=dev), ms <= 0

    def deriv(t, y, q):
        R, PR, _, PP = q
        X = torch.log(R) if log else R
        k = torch.clamp(torch.floor((X - X0) / h).long(), 0, p.n_grid - 2)
        x = X - (X0 + k.double() * h)
        c = ct[:, k]
        v = c[..., 0] + x * (c[..., 1] + x * (c[..., 2] + x * c[..., 3]))
        dv = (c[..., 1] + x * (2 * c[..., 2] + 3 * x * c[..., 3])) / (R if log else 1.0)
        ph = torch.polar(torch.ones_like(t * En), -(t * En))
        C = ph * y
        Cg = C[it]
        w = ((Gt @ v).view(D, N, B) * Cg).sum(0)
        u = ((Gt @ dv).view(D, N, B) * Cg).sum(0)
        pd = PP / (mu * R * R)
        Dw, Dy = ad * w[dn] - au * w[up], ad * y[dn] - au * y[up]
        f = -(C.conj() * u).real.sum(0) + PP * PP / (mu * R ** 3)
        return -1j * ph.conj() * w + 0.5 * pd * Dy, torch.stack([PR / mu, f, pd, (C.conj() * Dw).real.sum(0)])

    def step(A, q, steps, done):
        t = steps.double() * dt
        k1, l1 = deriv(t, A, q)
        k2, l2 = deriv(t + dt / 2, A + dt / 2 * k1, q + dt / 2 * l1)
        k3, l3 = deriv(t + dt / 2, A + dt / 2 * k2, q + dt / 2 * l2)
        k4, l4 = deriv(t + dt, A + dt * k3, q + dt * l3)
        An, qn = A + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4), q + dt / 6 * (l1 + 2 * l2 + 2 * l3 + l4)
        A, q = torch.where(done, A, An), torch.where(done, q, qn)
        steps = steps + (~done).long()
        return A, q, steps, done | ((q[0] >= rend) & (q[1] > 0)) | (steps >= ms)

    state = [A, q, steps, done]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step(*state)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for dst, new in zip(state, step(*state)):
            dst.copy_(new)
    for i in range(int(tr["max_steps"].max())):
        graph.replay()
        if i % 64 == 63 and bool(state[3].all()):
            break
    A = state[0].t().contiguous()
    return A.abs().square(), A


def _exact_rates(rs):
    dev = torch.device("cuda")
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    sig, g, E, U = T(rs.sigma), T(rs.g), T(rs.energy), [float(x) for x in rs.u]
    K, L = sig.shape[0], sig.shape[1]
    sym = 0.5 * (g[:, None] * sig + g[None, :] * sig.transpose(1, 2))
    S = np.zeros((K, K))  # second derivatives of the natural spline
    A, R = np.eye(K), np.zeros((K, K))
    for i in range(1, K - 1):
        h0, h1 = U[i] - U[i - 1], U[i + 1] - U[i]
        A[i, i - 1:i + 2] = [h0, 2 * (h0 + h1), h1]
        R[i, i - 1:i + 2] = [6 / h0, -6 / h0 - 6 / h1, 6 / h1]
    S = T(np.linalg.solve(A, R))
    x, w = np.polynomial.legendre.leggauss(16)
    x, w = T(0.5 * (x + 1.0)), T(0.5 * w)
    ia, ib = torch.triu_indices(L, L, device=dev)
    rate = torch.zeros((len(rs.kT), L, L), dtype=torch.float64, device=dev)
    P = 12
    cut = (torch.arange(P, device=dev, dtype=torch.float64) / P)[:, None]
    nodes = (cut + x[None] / P).reshape(-1)
    wts = (w / P).repeat(P)
    for a0 in range(0, len(ia), 100000):
        a, b = ia[a0:a0 + 100000], ib[a0:a0 + 100000]
        y = sym[:, a, b]
        M = S @ y
        dE = E[b] - E[a]
        u0 = 0.5 * dE.abs()
        for t, kT in enumerate(float(k) for k in rs.kT):
            acc = torch.zeros_like(u0)
            for k in range(-1, K - 1):
                lo = u0 if k < 0 else torch.clamp(u0, min=U[k])
                hi = torch.clamp(lo + 48.0 * kT, max=U[k + 1])
                wd = torch.clamp(hi - lo, min=0.0)
                V = lo[:, None] + wd[:, None] * nodes
                if k < 0:
                    f = (V - u0[:, None]) / (U[0] - u0)[:, None] * y[0][:, None]
                    wd = torch.where(u0 < U[0], wd, torch.zeros_like(wd))
                else:
                    h = U[k + 1] - U[k]
                    s = (V - U[k]) / h
                    r = 1.0 - s
                    f = r * y[k][:, None] + s * y[k + 1][:, None] + h * h / 6 * (
                        (r ** 3 - r) * M[k][:, None] + (s ** 3 - s) * M[k + 1][:, None])
                    f = f.clamp(min=0.0)
                one = (f * V * torch.exp(-(V - u0[:, None]) / kT)) @ wts * wd
                acc += torch.where(wd > 0, one, torch.zeros_like(one))
            yK, yJ = y[K - 1], y[K - 2]
            pw = torch.clamp(torch.log(yK / yJ) / math.log(U[K - 1] / U[K - 2]), -1.0, 0.0)
            pw = torch.where((yK > 0) & (yJ > 0), pw, torch.zeros_like(pw))
            s = 2.0 + pw
            top = torch.clamp(u0, min=U[K - 1])
            gam = torch.special.gammaincc(s, top / kT) * torch.exp(torch.lgamma(s) + u0 / kT)
            acc += yK * U[K - 1] ** (-pw) * kT ** s * gam
            c = math.sqrt(8.0 / (math.pi * rs.mu)) * kT ** -1.5 * acc
            rate[t, a, b] = c * torch.exp(-(0.5 * dE + u0) / kT) / g[a]
            rate[t, b, a] = c * torch.exp((0.5 * dE - u0) / kT) / g[b]
    return {"sigma_sym": sym, "rate": rate}


def exact(case, seed):
    kind = case["kind"]
    if kind == "rates":
        return _exact_rates(W.rate_set(n_levels=case["levels"], seed=seed,
                                       temps_k=tuple(np.geomspace(case["t_lo"], case["t_hi"], case["temps"]))))
    # the coupling algebra of the two molecules and of the asymmetric top, reverse-mode gradients and
    # adaptive steps have no short restatement
    if kind in ("mix", "adjoint") or case.get("rotor", "diatom") != "diatom" or case.get("tol"):
        return None
    p = _params(case)
    lmax = p.n_terms - 1
    rng_states = type("Labels", (), {"j": np.array([case["jmax"]]), "state": staticmethod(lambda j, m: j * j + j + m)})
    tr = _trajs(case, seed, [p.mu], _low_state(rng_states))
    per_step = 4 * (1.5e-4 + 4e-11 * p.n_states * len(tr) * (2 * lmax + 1))
    worst = min(int(tr["max_steps"].max()), int(2.2 * case["r0"] / (5.0 * math.sqrt(2.0 * float(W.cm(case["e_lo"])) / p.mu))))
    if worst * per_step > 11.0:
        return None
    log = kind == "sparse"
    pop, amp = _exact_diatom(case, p, tr, log=log, trunc=_trunc() if log else None)
    out = {"pop": pop, "ints": None}
    if case.get("host"):
        out = {"pop": pop, "amp": amp, "steps": None, "status": None}
    if case.get("precision") == "fp64":
        out["sigma"] = _exact_sigma(case, seed, p, pop, tr)
    return out


def _exact_sigma(case, seed, p, pop, tr):
    """sum over the trajectories of a group of weight * population of each level (level = j)"""
    group = np.random.default_rng(seed + 5).integers(0, SIGMA_GROUPS, case["n"])
    weight = 2.0 * np.pi * case["b_max"] * tr["b"] / case["n"]
    Wg = np.zeros((SIGMA_GROUPS, case["n"]))
    Wg[group, np.arange(case["n"])] = weight
    j = np.concatenate([np.full(2 * a + 1, a) for a in range(p.jmax + 1)])
    sel = np.zeros((len(j), p.jmax + 1))
    sel[np.arange(len(j)), j] = 1.0
    dev = pop.device
    return torch.from_numpy(Wg).to(dev) @ pop @ torch.from_numpy(sel).to(dev)
