"""The performance cases of the HEOM propagator: what a user has it do, through its public entry points.

A pass is one call as a user's program makes it: a whole propagation with its observables
(``heom.propagate_static``), a thermal state (``spectra.thermal_state``), the next steps of a run that the
program keeps on the GPU and the density matrix after them (``heom.Run``), one replay of a ragged batch
(``heom.Batch``) or one tick of a server's small requests (``heom.group_propagate``).  Hamiltonians,
dipoles and baths are drawn from the seed with the recipes of ``workloads.py``; ``exact`` states the same
propagation in plain torch, FP64, without the library.

``listed()`` holds the named cases, ``draw(rng)`` more of the same ranges:

  whole    2..16 sites, 0 or 1 mode per bath beyond the Drude mode, depth 2..6, workspace below 32 MiB
  thermal  2..9 sites, FP64, the state of every ADO
  run      2..24 sites, up to the 1,344,904 ADOs of the LHCII-like hierarchy; population runs (also from a
           coherence, whose ADOs are not Hermitian) and linear-absorption runs; every precision
  pulse    the two-exciton space of 2..7 sites (4..29 states) under a laser pulse
  batch    linear-absorption runs of many systems, three polarisations each
  group    population runs of many systems, mixed precision
"""
from __future__ import annotations

import math
from math import comb

import numpy as np
import torch

LHCII_WORK = comb(28 + 6, 6) * 14 ** 2  # elements of the largest hierarchy state


def _n_ado(sites, K, D):
    return comb(sites * (K + 1) + D, D)


# ---- the cases --------------------------------------------------------------------------------------


def listed():
    return [
        # the textbook check: a dimer's populations at every step (2000 steps of 1 fs), one small call
        dict(name="dimer-fp64", kind="whole", what="population", sites=2, K=0, D=4, precision="fp64",
             steps=2000, stride=1, dt=1.0, tau=50.0, T=300.0, start="site", poles="matsubara"),
        # population transfer in an FMO-sized complex (3060 ADOs) in FP64, recorded every 2 fs
        dict(name="fmo-population-fp64", kind="whole", what="population", sites=7, K=1, D=4, precision="fp64",
             steps=400, stride=4, dt=0.5, tau=166.0, T=77.0, start="site", poles="matsubara"),
        # one polarisation of the linear absorption of the same complex, mixed precision
        dict(name="fmo-absorption-mixed", kind="whole", what="absorption", sites=7, K=1, D=4, precision="fp32_mixed",
             steps=400, stride=4, dt=0.5, tau=166.0, T=77.0, start="site", poles="matsubara"),
        # the thermal state that emission spectra start from: every ADO comes back
        dict(name="fmo-thermal-fp64", kind="thermal", sites=7, K=1, D=3, steps=400, dt=1.0, tau=166.0, T=77.0,
             poles="matsubara"),
        # the large production run: an LHCII-sized hierarchy (1,344,904 ADOs of 14 x 14) advanced 10 fs, in
        # the precision for production and in FP64
        dict(name="lhcii-population-mixed", kind="run", what="population", sites=14, K=1, D=6,
             precision="fp32_mixed", steps=10, dt=1.0, tau=50.0, T=300.0, start="site", poles="matsubara"),
        dict(name="lhcii-population-fp64", kind="run", what="population", sites=14, K=1, D=6, precision="fp64",
             steps=4, dt=1.0, tau=50.0, T=300.0, start="site", poles="matsubara"),
        # linear absorption at the same size (15 states with the ground state)
        dict(name="lhcii-absorption-mixed", kind="run", what="absorption", sites=14, K=1, D=6,
             precision="fp32_mixed", steps=40, dt=1.0, tau=50.0, T=300.0, start="site", poles="matsubara"),
        # a mid-sized complex with an odd number of states above 16 (one ADO per warp)
        dict(name="sites19-population-mixed", kind="run", what="population", sites=19, K=0, D=5,
             precision="fp32_mixed", steps=20, dt=0.5, tau=90.0, T=300.0, start="site", poles="matsubara"),
        # pumped two-exciton space of the FMO-sized complex (29 states, 3060 ADOs), laser pulse, H(t)
        dict(name="two-exciton-pulse-fp64", kind="pulse", sites=7, K=1, D=4, precision="fp64", steps=10, dt=0.5,
             tau=166.0, T=77.0, poles="matsubara"),
        dict(name="two-exciton-pulse-mixed", kind="pulse", sites=7, K=1, D=4, precision="fp32_mixed", steps=20,
             dt=0.5, tau=166.0, T=77.0, poles="matsubara"),
        # the absorption of an ensemble of different complexes: 16 systems x 3 polarisations in one graph
        dict(name="ragged-batch-mixed", kind="batch", systems=16, n_max=16, precision="fp32_mixed", steps=20, dt=0.5),
        # a server's tick: 32 small requests of all sizes advance 50 steps together
        dict(name="serving-tick-mixed", kind="group", systems=32, n_max=24, steps=50, dt=0.5),
    ]


def _seconds(case):
    """A rough time of one pass, so that a drawn case costs no more than the largest listed one."""
    k = case["kind"]
    if k == "batch":
        return 0.01 * case["systems"] * case["steps"] / 20
    if k == "group":
        return 0.01 * case["systems"] * case["steps"] / 50
    n, fp64 = _n_ado(case["sites"], case["K"], case["D"]), case.get("precision", "fp64") == "fp64"
    if k == "pulse":
        N = 1 + case["sites"] + case["sites"] * (case["sites"] - 1) // 2
        return case["steps"] * (1e-4 + n * N ** 3 * (1.2e-10 if fp64 else 1.2e-11))
    N = case["sites"] + (case.get("what") == "absorption")
    per = n * N ** (1 if case.get("what") == "absorption" else 2) * (2e-9 if fp64 else 2.5e-11 * N ** 0.5)
    if case.get("start") == "coherence":
        per *= 3
    return case["steps"] * (2e-4 + per * (2 if case.get("what") == "absorption" else 1))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    while True:
        kind = rng.choice(["whole", "whole", "run", "run", "run", "thermal", "pulse", "batch", "group"])
        c = dict(kind=kind)
        if kind == "batch":
            c.update(systems=_log_int(rng, 2, 16), n_max=rng.randint(8, 16),
                     precision=rng.choice(["fp32_mixed", "fp32_mixed", "fp64"]), steps=_log_int(rng, 5, 30), dt=0.5)
            return c
        if kind == "group":
            c.update(systems=_log_int(rng, 2, 40), n_max=rng.randint(8, 24), steps=_log_int(rng, 10, 60), dt=0.5)
            return c
        c.update(K=rng.randint(0, 1), D=rng.randint(2, 6), dt=rng.choice([0.25, 0.5]),
                 tau=round(rng.uniform(50.0, 200.0), 1), T=rng.choice([77.0, 300.0]),
                 poles=rng.choice(["matsubara", "matsubara", "pade"]))
        if kind == "pulse":
            c.update(sites=rng.randint(2, 7), D=rng.randint(2, 4), precision=rng.choice(["fp64", "fp32_mixed"]),
                     steps=_log_int(rng, 5, 100))
            N = 1 + c["sites"] + c["sites"] * (c["sites"] - 1) // 2
        elif kind == "thermal":
            c.update(sites=rng.randint(2, 9), D=rng.randint(2, 4), steps=_log_int(rng, 50, 800))
            N = c["sites"]
        else:
            what = rng.choice(["population", "population", "absorption"])
            prec = rng.choice(["fp64", "fp32_mixed", "fp32_mixed"])
            if kind == "whole":
                c.update(what=what, sites=rng.randint(2, 16), precision=prec, steps=_log_int(rng, 50, 2000),
                         stride=rng.choice([1, 2, 5]), start="site")
            else:
                start = rng.choice(["site", "site", "site", "coherence"]) if what == "population" else "site"
                if what == "population" and start == "site":
                    prec = rng.choice(["fp64", "fp32_mixed", "fp32_mixed", "split_tf32"])
                c.update(what=what, sites=rng.randint(2, 24 if what == "population" else 23), precision=prec,
                         steps=_log_int(rng, 2, 100), start=start)
            N = c["sites"] + (what == "absorption")
        n = _n_ado(c["sites"], c["K"], c["D"])
        per = N if c.get("what") == "absorption" else N * N
        bytes_el = 16 if c.get("precision", "fp64") == "fp64" else 8
        if kind == "whole":  # the static workspace: three copies and the link records
            room = n * (3 * per * bytes_el + 64 * min(c["D"] + c["sites"] * (c["K"] + 1), 40)) + 4096 * 30 * 8
            if room > 24 << 20:
                continue
        if n * per > LHCII_WORK or n > 3_000_000 or (kind in ("thermal", "pulse") and n > 8000) or _seconds(c) > 0.2:
            continue
        return c


# ---- inputs: the recipes of the repository's workloads, drawn from the seed --------------------------


def _site_system(rng, sites, K, D, tau, T, lam=None, poles="matsubara"):
    from paper_1803_03498_gb300 import workloads as wl

    H = np.zeros((sites, sites))
    H[np.diag_indices(sites)] = rng.uniform(12100.0, 12600.0, sites)
    iu = np.triu_indices(sites, 1)
    H[iu] = rng.normal(0.0, 40.0, len(iu[0]))
    H = H + np.triu(H, 1).T
    lam = [35.0] * sites if lam is None else lam
    tau = [tau] * sites if np.isscalar(tau) else tau
    return wl.System(f"{sites} sites K={K} D={D}", H, list(range(sites)), lam, tau, [T] * sites, K=K, D=D,
                     decomposition=poles)


def _random_baths(rng, n):
    return list(rng.uniform(20.0, 100.0, n)), list(rng.uniform(50.0, 200.0, n)), float(rng.choice([77.0, 300.0]))


def _propagations(case, seed):
    """The propagations of a case, and its laser pulse (or None)."""
    from paper_1803_03498_gb300 import workloads as wl

    rng = np.random.default_rng([seed, 1803])
    kind = case["kind"]
    if kind == "batch":
        # the sizes are the case's (the same for every seed), the numbers in them the seed's
        sizes, props = np.random.default_rng(case["systems"] * 100 + case["n_max"]), []
        for _ in range(case["systems"]):
            n, D, K = int(sizes.integers(2, case["n_max"] + 1)), int(sizes.integers(3, 6)), int(sizes.integers(0, 2))
            lam, tau, T = _random_baths(rng, n)
            s = _site_system(rng, n, K, D, tau, T, lam)
            props += wl.dipole_runs(s, wl.unit_dipoles(rng, n), case["dt"], case["steps"], "batch")
        return props, None
    if kind == "group":
        sizes, props = np.random.default_rng(case["systems"] * 100 + case["n_max"] + 7), []
        while len(props) < case["systems"]:
            n, D, K = int(sizes.integers(2, case["n_max"] + 1)), int(sizes.integers(2, 7)), int(sizes.integers(0, 2))
            if _n_ado(n, K, D) > 50_000 or _n_ado(n, K, D) * n * n > 4e6:  # what a server batches
                continue
            lam, tau, T = _random_baths(rng, n)
            s = _site_system(rng, n, K, D, tau, T, lam)
            re = np.zeros((n, n))
            re[0, 0] = 1.0
            props.append(wl.Propagation(s, re, np.zeros((n, n)), case["dt"], case["steps"]))
        return props, None
    s = _site_system(rng, case["sites"], case["K"], case["D"], case["tau"], case["T"], poles=case["poles"])
    n = s.N
    if kind == "pulse":
        g, _ = wl.two_exciton(s)
        mup = wl.two_exciton_dipole(n, wl.unit_dipoles(rng, n)[:, 0])
        re = np.zeros((g.N, g.N))
        re[0, 0] = 1.0
        p = wl.Propagation(g, re, np.zeros_like(re), case["dt"], case["steps"])
        return [p], wl.Pulse(mup, 60.0, 10.0, 15.0, phase=0.4, detuning_cm=30.0)
    if kind != "thermal" and case["what"] == "absorption":
        p = wl.dipole_runs(s, wl.unit_dipoles(rng, n), case["dt"], case["steps"], "absorption")[0]
        p.system.decomposition = case["poles"]
        return [p], None
    re, im = np.zeros((n, n)), np.zeros((n, n))
    if case.get("start") == "coherence":  # |psi><1| of a superposition: not Hermitian
        re[:, 0], im[:, 0] = rng.normal(size=n), rng.normal(size=n)
    else:
        re[0, 0] = 1.0
    return [wl.Propagation(s, re, im, case["dt"], case["steps"])], None


def prepare(case, seed):
    from paper_1803_03498_gb300 import heom

    props, pulse = _propagations(case, seed)
    kind, state = case["kind"], {"case": case, "props": props}
    if kind == "whole":  # the hierarchy is the plan that a program keeps for its calls
        s = props[0].system
        state["hier"] = heom.Hierarchy(s.n_modes, s.D)
    elif kind != "thermal":
        hier = {}
        state["runs"] = []
        for p in props:
            key = (p.system.n_modes, p.system.D)
            if key not in hier:
                hier[key] = heom.Hierarchy(*key)
            state["runs"].append(heom.Run(p.system, p.rho0_re, p.rho0_im, precision=case.get("precision", "fp32_mixed"),
                                          w=p.w, max_records=2, hier=hier[key], time_dependent=pulse is not None))
        if pulse is not None:
            state["runs"][0].set_field(pulse)
        if kind == "batch":
            state["batch"] = heom.Batch(state["runs"], case["dt"], case["steps"], obs_stride=0)
    return state


def run(state):
    from paper_1803_03498_gb300 import heom, spectra

    c, p = state["case"], state["props"][0]
    if c["kind"] == "whole":
        obs, rho = heom.propagate_static(p.system, p.rho0_re, p.rho0_im, precision=c["precision"], w=p.w, dt_fs=c["dt"],
                                         n_steps=c["steps"], obs_stride=c["stride"], hier=state["hier"])
        return {"records": obs, "rho": rho}
    if c["kind"] == "thermal":
        re, im, resid = spectra.thermal_state(p.system, c["dt"], c["steps"])
        return {"re": re, "im": im, "resid": resid}
    runs = state["runs"]
    if c["kind"] == "batch":
        state["batch"].launch()
    elif c["kind"] == "group":
        heom.group_propagate(runs, c["dt"], c["steps"])
    else:
        runs[0].propagate(c["dt"], c["steps"])
        if c["precision"] == "fp64":  # rho and the first level, the moments of the baths
            re, im = runs[0].get_ados(0, 1 + p.system.n_modes)
            return {"re": re, "im": im}
        return {"rho": runs[0].sigma0()}
    return {"rho": np.concatenate([r.sigma0().ravel() for r in runs])}


def work(case):
    """Per RK4 step four evaluations of the right-hand side, each of which reads the state and writes the
    result.  A Hermitian ADO holds N^2 real numbers, a general one 2 N^2, an ADO of a linear-absorption
    run 2 N.  Operations: the commutator (half of it, 4 N^3 with a real H, for Hermitian ADOs), decay and
    combination, and the linked rows."""
    props, pulse = _propagations(case, 0)
    total = {"bytes": 0.0, "flops": 0.0}
    for p in props:
        s = p.system
        n, N, M, D = s.n_ado, s.N, s.n_modes, s.D
        links = 2.0 * M * comb(M + D - 1, D - 1) if D > 0 else 0.0  # one down and one up per (ADO, mode)
        column = p.w is not None
        general = case.get("start") == "coherence"
        size = 8.0 if case.get("precision", "fp64") == "fp64" and case["kind"] != "group" else 4.0
        if column:
            reals, flops = 2.0 * N, n * (4.0 * N * N + 8.0 * N) + 8.0 * links
        elif pulse is not None:  # complex H(t); every coupling acts on the states that hold its site
            reals, flops = N * N, n * (8.0 * N ** 3 + 8.0 * N * N) + links * case["sites"] * 8.0 * N
        else:
            reals = N * N * (2.0 if general else 1.0)
            flops = n * ((8.0 if general else 4.0) * N ** 3 + 8.0 * N * N) + links * 8.0 * N * (2.0 if general else 1.0)
        total["bytes"] += 4 * case["steps"] * n * 2 * reals * size
        total["flops"] += 4 * case["steps"] * flops
    return total


# ---- the same propagation in plain torch, FP64 --------------------------------------------------------

_TWO_PI_C, _KB = 2.0 * math.pi * 2.99792458e-5, 0.6950348004  # rad/fs per cm^-1, cm^-1 per K


def _modes(s):
    """Rates, coefficients, lambda nu of every mode and the terminator rate of every bath, rad/fs."""
    K, gam, c, lnu, delta = s.K, [], [], [], []
    if s.decomposition == "pade" and K > 0:
        m = np.arange(1, 2 * K)
        e1 = 1.0 / np.sqrt((2.0 * m + 1) * (2.0 * m + 3))
        m = np.arange(1, 2 * K - 1)
        e2 = 1.0 / np.sqrt((2.0 * m + 3) * (2.0 * m + 5))
        top = lambda e, k: 2.0 / np.sort(np.linalg.eigvalsh(np.diag(e, 1) + np.diag(e, -1)))[::-1][:k]  # noqa: E731
        xi, zeta = top(e1, K), top(e2, K - 1) if K > 1 else np.zeros(0)
        eta = [0.5 * K * (2 * K + 3) * np.prod(zeta ** 2 - x * x) / np.prod([y * y - x * x for y in xi if y != x])
               for x in xi]
    for lam, tau, T in zip(s.lambda_cm, s.tau_fs, s.T_K):
        lam, nu, beta = _TWO_PI_C * lam, 1.0 / tau, 1.0 / (_TWO_PI_C * _KB * T)
        if s.decomposition == "pade":
            g = [xi[k] / beta for k in range(K)]
            cs = [4.0 * lam * nu * eta[k] * g[k] / (beta * (g[k] ** 2 - nu * nu)) for k in range(K)]
            c0 = 2.0 * lam / beta * (1.0 - sum(2.0 * eta[k] * nu * nu / (g[k] ** 2 - nu * nu) for k in range(K)))
        else:
            g = [2.0 * math.pi * (k + 1) / beta for k in range(K)]
            cs = [4.0 * lam * nu / beta * x / (x * x - nu * nu) for x in g]
            c0 = lam * nu / math.tan(0.5 * beta * nu)
        gam += [nu] + g
        c += [c0] + cs
        lnu += [lam * nu] + [0.0] * K
        delta.append(2.0 * lam / (beta * nu) - sum(x / y for x, y in zip([c0] + cs, [nu] + g)))
    return np.array(gam), np.array(c), np.array(lnu), np.array(delta)


def _hierarchy(M, D, dev):
    """Occupations [n_ado, M] and, per mode, the index of the ADO with one more (-1: none), level by
    level, inside a level by the colexicographic rank of the bars b_j = (j - 1) + n_1 + ... + n_j."""
    binom = torch.tensor([[comb(a, j) for j in range(M + 1)] for a in range(M + D + 1)], dtype=torch.int64, device=dev)
    js = torch.arange(1, M, device=dev)
    first = torch.tensor([comb(M + L - 1, M) if L else 0 for L in range(D + 2)], dtype=torch.int64, device=dev)

    def rank(b, level):  # b [n, M - 1]
        u = first[level].clone()
        for q in range(M - 1):
            u += binom[b[:, q], q + 1]
        return u

    n = torch.zeros((1, M), dtype=torch.int64, device=dev)
    every = [n]
    for L in range(1, D + 1):  # each ADO of the level below with one more in a mode at or after its last
        last = torch.where(n > 0, torch.arange(M, device=dev), 0).amax(1)
        up = torch.repeat_interleave(M - last, 1)
        src = torch.repeat_interleave(torch.arange(n.shape[0], device=dev), up)
        at = torch.arange(src.shape[0], device=dev) - (torch.cumsum(up, 0) - up)[src] + last[src]
        m = n[src].clone()
        m[torch.arange(m.shape[0], device=dev), at] += 1
        u = rank(js - 1 + torch.cumsum(m, 1)[:, :-1], torch.full((m.shape[0],), L, device=dev))
        n = m[torch.argsort(u)]
        every.append(n)
    n = torch.cat(every)
    level = n.sum(1)
    bars = js - 1 + torch.cumsum(n, 1)[:, :-1]
    low = torch.nonzero(level < D)[:, 0]
    plus = []
    for l in range(M):
        b = bars[low].clone()
        b[:, l:] += 1
        plus.append(rank(b, level[low] + 1))
    return n, low, plus


class _Exact:
    """Eq. HEOM, element by element, on every ADO: the full matrices, or (columns) column 0 of runs that
    stay in it."""

    def __init__(self, s, columns=False):
        self.dev = dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        gam, c, lnu, delta = _modes(s)
        N, M, K1 = s.N, s.n_modes, s.K + 1
        H = np.array(s.H, dtype=float)
        self.H0 = H - np.eye(N) * 0.5 * (H.diagonal().max() + H.diagonal().min())
        self.H = torch.tensor(_TWO_PI_C * self.H0, device=dev)
        self.Hc = None  # H(t) of a laser field
        mask = np.zeros((len(s.bath_state), N))
        if s.bath_mask is not None:
            mask[:] = s.bath_mask
        else:
            mask[np.arange(len(s.bath_state)), s.bath_state] = 1.0
        term = sum(d * (m[:, None] - m[None, :]) ** 2 for d, m in zip(delta, mask))
        n, low, plus = _hierarchy(M, s.D, dev)
        self.n_ado, self.N, self.columns = n.shape[0], N, columns
        self.g = n.double() @ torch.tensor(gam, device=dev)
        to, frm, st, R = [], [], [], []
        for l in range(M):
            ac = abs(c[l])
            nl = n[low, l].double()
            hi = plus[l]
            r_up = 1j * torch.sqrt((nl + 1) * ac)
            r_dn = torch.sqrt((nl + 1) / ac) * complex(lnu[l], c[l])
            for state in np.nonzero(mask[l // K1])[0]:
                for a, b, r in ((low, hi, r_up), (hi, low, r_dn)):
                    to.append(a)
                    frm.append(b)
                    st.append(torch.full_like(a, int(state)))
                    R.append(r)
        self.to, self.frm, self.st = torch.cat(to), torch.cat(frm), torch.cat(st)
        self.R = torch.cat(R).to(torch.complex128)
        self.T = torch.tensor(term, device=dev)
        if columns:
            self.T = self.T[:, 0]

    def rhs(self, S):
        N, real = self.N, torch.view_as_real
        H = self.H.to(torch.complex128) if self.Hc is None else self.Hc
        if self.columns:  # S [n, N]
            out = -1j * (S @ H.T) + 1j * self.H[0, 0] * S - (self.g[:, None] + self.T) * S
            out = out.reshape(-1)
            add = self.R * S.reshape(-1)[self.frm * N + self.st]
            real(out).index_add_(0, self.to * N + self.st, real(add))
            return out.reshape(-1, N)
        out = (S.reshape(-1, N) @ (1j * H)).reshape(S.shape)
        out -= torch.matmul(1j * H, S)
        out -= (self.g[:, None, None] + self.T) * S
        col = torch.zeros_like(S)
        out_r, col_r = real(out).view(-1, 2 * N), real(col).view(-1, 2 * N)
        rows = S.reshape(-1, N)
        St = S.transpose(1, 2)
        for a in range(0, self.to.shape[0], 1 << 21):
            q = slice(a, a + (1 << 21))
            at = self.to[q] * N + self.st[q]
            out_r.index_add_(0, at, real(self.R[q, None] * rows[self.frm[q] * N + self.st[q]]).reshape(-1, 2 * N))
            col_r.index_add_(0, at, real(self.R[q].conj()[:, None] * St[self.frm[q], self.st[q]]).reshape(-1, 2 * N))
        out += col.transpose(1, 2)
        return out

    def field(self, pulse, t):
        x = (t - pulse.t_center_fs) / pulse.sigma_fs
        g = _TWO_PI_C * pulse.amp_cm * np.exp(-0.5 * x * x - 1j * (_TWO_PI_C * pulse.detuning_cm * t + pulse.phase))
        self.Hc = torch.tensor(_TWO_PI_C * self.H0 - g * pulse.mu_plus - np.conj(g) * pulse.mu_plus.T, device=self.dev)

    def propagate(self, S, h, steps, stride=0, pulse=None):
        """Classic RK4; the root ADO after every stride steps, the start first."""
        seen = [S[0].clone()]
        for k in range(steps):
            t = k * h
            if pulse is not None:
                self.field(pulse, t)
            k1 = self.rhs(S)
            acc = S + h / 6 * k1
            if pulse is not None:
                self.field(pulse, t + h / 2)
            k1 = self.rhs(S + h / 2 * k1)
            acc += h / 3 * k1
            k1 = self.rhs(S + h / 2 * k1)
            acc += h / 3 * k1
            if pulse is not None:
                self.field(pulse, t + h)
            S = acc + h / 6 * self.rhs(S + h * k1)
            if stride and (k + 1) % stride == 0:
                seen.append(S[0].clone())
        return S, seen


def _exact_seconds(case, props):
    total = 0.0
    for p in props:
        s, N = p.system, p.system.N
        column = p.w is not None
        links = 2.0 * s.n_modes * comb(s.n_modes + s.D - 1, s.D - 1) * (case["sites"] if case["kind"] == "pulse" else 1)
        moved = s.n_ado * N * (1 if column else N) * 16 * 12 + links * (96 if column else 200 * N)
        flops = 0 if column else s.n_ado * 16.0 * N ** 3
        total += 4 * case["steps"] * (4e-4 + moved / 2e12 + flops / 4e11)
    return total


def exact(case, seed):
    props, pulse = _propagations(case, seed)
    if _exact_seconds(case, props) > 15.0:
        return None
    rhos = []
    for p in props:
        s, column = p.system, p.w is not None
        e = _Exact(s, column)
        S = torch.zeros((e.n_ado, e.N) if column else (e.n_ado, e.N, e.N), dtype=torch.complex128, device=e.dev)
        if case["kind"] == "thermal":
            H0 = np.array(s.H, dtype=float) - np.diag(s.lambda_cm)
            w, U = np.linalg.eigh(H0)
            q = np.exp(-(w - w.min()) / (_KB * s.T_K[0]))
            rho = (U * (q / q.sum())) @ U.T
            S[0] = torch.tensor(0.5 * (rho + rho.T), device=e.dev)
        else:
            rho = torch.tensor(p.rho0_re + 1j * p.rho0_im, device=e.dev)
            S[0] = rho[:, 0] if column else rho
        S, seen = e.propagate(S, case["dt"], case["steps"], case.get("stride", 0), pulse)
        if case["kind"] == "thermal":
            L = e.rhs(S)
            resid = float(torch.linalg.vector_norm(L) / torch.linalg.vector_norm(S))
            return {"re": S.real.cpu().numpy(), "im": S.imag.cpu().numpy(), "resid": resid}
        if case["kind"] in ("run", "pulse") and case["precision"] == "fp64":
            top = S[: 1 + s.n_modes]
            if column:
                full = torch.zeros(top.shape + (e.N,), dtype=top.dtype, device=e.dev)
                full[:, :, 0] = top
                top = full
            return {"re": top.real.cpu().numpy(), "im": top.imag.cpu().numpy()}
        if case["kind"] == "whole":
            seen = torch.stack(seen).cpu().numpy()
            rec = np.zeros((len(seen), e.N + 5))
            if column:
                corr = seen @ p.w
                rec[:, e.N + 2], rec[:, e.N + 3] = corr.real, corr.imag
                rec[:, e.N + 4] = np.abs(seen).max(1)
            else:
                d = np.diagonal(seen, axis1=1, axis2=2)
                rec[:, : e.N], rec[:, e.N], rec[:, e.N + 1] = d.real, d.real.sum(1), d.imag.sum(1)
                rec[:, e.N + 4] = np.abs(seen - seen.conj().transpose(0, 2, 1)).max((1, 2))
        rho = S[0].cpu().numpy()
        if column:
            full = np.zeros((e.N, e.N), dtype=complex)
            full[:, 0] = rho
            rho = full
        if case["kind"] == "whole":
            return {"records": rec, "rho": rho}
        rhos.append(rho if case["kind"] in ("run", "pulse") else rho.ravel())
        del e, S
    return {"rho": rhos[0] if case["kind"] in ("run", "pulse") else np.concatenate(rhos)}
