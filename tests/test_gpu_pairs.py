"""The element kernels (csrc/resident.cuh, csrc/lean.cuh) at the sizes where they can go wrong: one state, the last size
of each form (8 and 9, where the commutator of a small part turns to fixed point; 22 and 23, where one ADO's pairs fill a
CTA), one ADO, chunks that do not fill, non-Hermitian and complex runs; launches of whole steps against launches of
single stages; and the ends of the exponent range, where the fixed-point commutator gives way to FMAs."""
import numpy as np
import pytest

from helpers import oracle_for, oracle_propagate
from paper_1803_03498_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def heom():
    from paper_1803_03498_gb300.build import build
    build()
    from paper_1803_03498_gb300 import heom as h
    h.load()
    return h


def _prop(N, K, D, start="site", cplx=False):
    rng = np.random.default_rng(1803300 + N)
    H = np.diag(rng.uniform(0.0, 400.0, N)) + np.triu(rng.normal(0.0, 40.0, (N, N)), 1)
    H = H + np.triu(H, 1).T
    if cplx:
        A = np.triu(rng.normal(0.0, 20.0, (N, N)), 1)
        H = H + 1j * (A - A.T)
    s = wl.System(f"N={N}", H, list(range(N)), [35.0] * N, [60.0] * N, [300.0] * N, K=K, D=D)
    re, im = np.zeros((N, N)), np.zeros((N, N))
    if start == "site":
        re[0, 0] = 1.0
    else:
        re[:, 0], im[:, 0] = rng.normal(size=N), rng.normal(size=N)
    return wl.Propagation(s, re, im, 0.5, 21)


CASES = [(1, 1, 2, "site", False), (2, 0, 0, "site", False), (2, 0, 6, "site", False), (5, 1, 4, "site", False),
         (8, 1, 2, "site", False), (9, 0, 3, "site", False), (14, 1, 2, "site", False), (16, 0, 3, "site", False),
         (22, 0, 2, "site", False), (23, 0, 2, "site", False), (24, 0, 1, "site", False), (7, 1, 3, "coherence", False),
         (18, 0, 2, "coherence", False), (6, 1, 2, "site", True), (12, 0, 2, "coherence", True)]


@pytest.mark.parametrize("N,K,D,start,cplx", CASES)
def test_fp64_elements_match_oracle(heom, N, K, D, start, cplx):
    """Every element of every ADO after 21 steps within 1e-12 of the oracle (relative to the largest where that is
    above 1), whole steps per launch and single stages (kernel timing on) bit for bit alike."""
    p = _prop(N, K, D, start, cplx)
    m, ore, oim, oobs = oracle_propagate(p, p.n_steps, stride=4)
    ref = ore + 1j * oim
    got = []
    for timing in (False, True):
        r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision="fp64", max_records=8)
        r.set_timing(timing)
        r.propagate(p.dt_fs, p.n_steps, 4)
        re, im = r.get_ados(0, r.n_ado)
        got.append((re + 1j * im, r.observables()))
        r.close()
    assert np.max(np.abs(got[0][0] - ref)) <= 1e-12 * max(1.0, np.max(np.abs(ref)))
    assert np.max(np.abs(got[0][1][:, :N + 4] - oobs)) <= 1e-12 * max(1.0, np.max(np.abs(oobs)))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("N,K,D,start", [(2, 0, 4, "site"), (7, 1, 3, "site"), (14, 1, 2, "site"), (22, 0, 2, "site"),
                                         (23, 0, 2, "site"), (10, 0, 1, "site"), (7, 1, 3, "coherence")])
def test_mixed_whole_steps_equal_stages(heom, N, K, D, start):
    """Mixed runs: whole steps per launch and single stages give the same bits in every ADO and record, and the
    populations stay within 1e-6 of the oracle (D = 1: no FP32 body)."""
    p = _prop(N, K, D, start)
    m, ore, oim, oobs = oracle_propagate(p, p.n_steps, stride=3)
    got = []
    for timing in (False, True):
        r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision="fp32_mixed", max_records=9)
        r.set_timing(timing)
        r.propagate(p.dt_fs, p.n_steps, 3)
        got.append((r.get_ados(0, r.n_ado), r.observables()))
        r.close()
    assert np.max(np.abs(got[0][1][:, :N] - oobs[:, :N])) <= 1e-6 * max(1.0, np.max(np.abs(oobs)))
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0][0], got[1][0][0]) and np.array_equal(got[0][0][1], got[1][0][1])


def test_whole_steps_on_several_streams(heom):
    """Launches of whole steps from four threads, each on a stream of its own, give what each run gives alone."""
    import threading

    import torch

    props = [_prop(7, 1, 3), _prop(14, 1, 2), _prop(5, 1, 4), _prop(9, 0, 3)]
    kinds = ["fp64", "fp32_mixed", "fp64", "fp32_mixed"]

    def go(p, kind, stream):
        with torch.cuda.stream(stream):
            r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision=kind, max_records=2)
            for _ in range(3):
                r.propagate(p.dt_fs, 150, 0)
            out = r.get_ados(0, r.n_ado)
            r.close()
            return out

    alone = [go(p, k, torch.cuda.Stream()) for p, k in zip(props, kinds)]
    got = [None] * 4

    def work(i):
        got[i] = go(props[i], kinds[i], torch.cuda.Stream())

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    for a, b in zip(alone, got):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("N", [9, 14])
@pytest.mark.parametrize("scale", [1.0, 1e-150, 1e-285, 1e-320, 1e285])
def test_fixed_point_commutator_scales(heom, N, scale):
    """One right-hand side of a dense Hermitian state times a power of ten (the smallest a subnormal, the largest near
    the end of the range) equals the oracle's of the unscaled state times the same: 1e-14 of the largest element, plus
    the spacing of subnormals times the number of terms."""
    p = _prop(N, 0, 2)
    m = oracle_for(p.system)
    rng = np.random.default_rng(N)
    x = rng.standard_normal((m.n_ado, N, N)) + 1j * rng.standard_normal((m.n_ado, N, N))
    x = 0.5 * (x + np.conj(np.transpose(x, (0, 2, 1)))) * 10.0 ** rng.uniform(-12, 0, (m.n_ado, 1, 1))
    x[3] = 0
    xs = (x.real * scale) + 1j * (x.imag * scale)
    ore, oim = m.rhs(np.ascontiguousarray(x.real), np.ascontiguousarray(x.imag))
    r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision="fp64", max_records=2)
    r.set_ados(0, xs.real, xs.imag)
    gre, gim = r.rhs_eval(0, m.n_ado)
    r.close()
    ref = ore * scale + 1j * (oim * scale)
    assert np.max(np.abs(gre + 1j * gim - ref)) <= 1e-14 * np.max(np.abs(ref)) + 200 * 5e-324


def test_non_finite_elements_stay_visible(heom):
    """An Inf or NaN in one ADO makes that ADO's right-hand side non-finite and leaves unlinked ADOs finite."""
    p = _prop(14, 0, 2)
    m = oracle_for(p.system)
    rng = np.random.default_rng(3)
    x = rng.standard_normal((m.n_ado, 14, 14))
    x = 0.5 * (x + np.transpose(x, (0, 2, 1)))
    for bad in (np.inf, np.nan):
        y = x.copy()
        y[0, 2, 2] = bad
        r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision="fp64", max_records=2)
        r.set_ados(0, y, np.zeros_like(y))
        gre, gim = r.rhs_eval(0, m.n_ado)
        r.close()
        assert not np.all(np.isfinite(gim[0]))
        assert np.all(np.isfinite(gre[15:])) and np.all(np.isfinite(gim[15:]))  # level 2: no link to the root


@pytest.mark.parametrize("sites,K,D,precision", [(1, 1, 3, "fp64"), (2, 0, 6, "fp32_mixed"), (7, 1, 3, "fp32_mixed"),
                                                 (7, 1, 2, "fp64"), (9, 1, 1, "fp32_mixed"), (16, 0, 3, "fp32_mixed"),
                                                 (23, 0, 2, "fp32_mixed"), (23, 0, 2, "fp64"), (5, 2, 2, "fp64")])
def test_column_whole_steps_equal_stages(heom, sites, K, D, precision):
    """Column-0 runs: whole steps per launch and single stages (kernel timing on) give the same bits in every record
    and ADO; FP64 within 1e-12 of the oracle, mixed correlations within 1e-5 of it (K = 2: up to six records per
    state, D = 1: no FP32 body)."""
    rng = np.random.default_rng(1803400 + sites)
    H = np.diag(rng.uniform(0.0, 400.0, sites)) + np.triu(rng.normal(0.0, 40.0, (sites, sites)), 1)
    s = wl.System(f"{sites} sites", H + np.triu(H, 1).T, list(range(sites)), [35.0] * sites, [60.0] * sites,
                  [300.0] * sites, K=K, D=D)
    p = wl.dipole_runs(s, wl.unit_dipoles(rng, sites), 0.5, 23, "col")[0]
    m, ore, oim, oobs = oracle_propagate(p, p.n_steps, stride=5)
    got = []
    for timing in (False, True):
        r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision=precision, w=p.w, max_records=8)
        assert r.layout() == 1
        r.set_timing(timing)
        r.propagate(p.dt_fs, p.n_steps, 5)
        got.append((r.get_ados(0, r.n_ado), r.observables()))
        r.close()
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0][0], got[1][0][0]) and np.array_equal(got[0][0][1], got[1][0][1])
    N = sites + 1
    tol = (1e-12 if precision == "fp64" else 1e-5) * max(1.0, np.max(np.abs(oobs)))
    assert np.max(np.abs(got[0][1][:, :N + 4] - oobs)) <= tol
    if precision == "fp64":
        assert np.max(np.abs(got[0][0][0] + 1j * got[0][0][1] - (ore + 1j * oim))) <= tol
