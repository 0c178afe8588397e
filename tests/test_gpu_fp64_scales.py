"""FP64 kernels over orders of magnitude, ADO by ADO: hierarchies whose ADOs differ by twelve decades, scaled towards both
ends of the exponent range, and Inf and NaN.  Every ADO's right-hand side is held to the rounding of its own operands (its
own tile and its neighbours'), so that another ADO's scale or a lost small ADO shows.  The cases reach every FP64
kernel: the pair kernels (9, 18, 22 states), the element kernels (23 states, complex H, not Hermitian, general runs) and
the column kernel at each of its sizes, in hierarchies above the line where it takes over from whole-step launches."""
import numpy as np
import pytest

from helpers import oracle_for, oracle_propagate
from paper_1803_03498_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CM = 2.0 * np.pi * 2.99792458e-5  # rad/fs per cm^-1


@pytest.fixture(scope="module")
def heom():
    from paper_1803_03498_gb300.build import build
    build()
    from paper_1803_03498_gb300 import heom as h
    h.load()
    return h


def _system(N, D, cplx=False):
    rng = np.random.default_rng(1803700 + N)
    H = np.diag(rng.uniform(0.0, 400.0, N)) + np.triu(rng.normal(0.0, 40.0, (N, N)), 1)
    H = H + np.triu(H, 1).T
    if cplx:
        A = np.triu(rng.normal(0.0, 20.0, (N, N)), 1)
        H = H + 1j * (A - A.T)
    return wl.System(f"N={N}", H, list(range(N)), [35.0] * N, [60.0] * N, [300.0] * N, K=0, D=D)


def _run(heom, s, general=False):
    rho = np.zeros((s.N, s.N))
    rho[0, 0] = 1.0
    return heom.Run(s, rho, np.zeros_like(rho), precision="fp64", max_records=8, time_dependent=general)


COLUMN = [(8, 8), (9, 9), (10, 7), (11, 7), (12, 6), (13, 6), (14, 6), (15, 6), (16, 4)]
# (states, depth, Hermitian, complex H, general)
CASES = [(9, 2, True, False, False), (18, 2, True, False, False), (22, 2, True, False, False), (23, 2, True, False, False),
         (12, 2, False, False, False), (6, 3, True, True, False), (9, 2, False, True, False), (9, 2, True, False, True)]


def _state(rng, n_ado, N, herm):
    x = rng.standard_normal((n_ado, N, N)) + 1j * rng.standard_normal((n_ado, N, N))
    if herm:
        x = 0.5 * (x + np.conj(np.transpose(x, (0, 2, 1))))
    x *= 10.0 ** rng.uniform(-12, 0, (n_ado, 1, 1))
    x[3] = 0.0
    x[5, :, 1] = x[5, 1, :] = 0.0  # a zero column (and row)
    return x


def _check(heom, N, D, herm, cplx, general, scale):
    s = _system(N, D, cplx)
    m = oracle_for(s)
    rng = np.random.default_rng(N)
    x = _state(rng, m.n_ado, N, herm)
    r = _run(heom, s, general)
    r.set_ados(0, x.real * scale, x.imag * scale)
    gre, gim = r.rhs_eval(0, m.n_ado)
    _, plus, minus = r.hier.export()
    r.close()
    us = np.unique(np.concatenate([np.arange(min(8, m.n_ado)), [m.n_ado - 1], rng.integers(0, m.n_ado, 200)]))
    ore, oim = m.rhs_list(us, np.ascontiguousarray(x.real), np.ascontiguousarray(x.imag))
    modes = heom.bath_modes(s)
    ac = np.abs(modes["c"])
    link = np.sqrt(D + 1.0) * np.max(np.sqrt(ac) + np.abs(modes["lamnu"] + 1j * modes["c"]) / np.sqrt(ac))
    rates = D * modes["gamma"].max() + 2.0 * np.abs(modes["term"]).max()
    top = np.abs(x).max((1, 2))
    near = np.concatenate([plus, minus], 1)[us].astype(np.int64)
    m_u = np.maximum(top[us], np.where(near >= 0, top[np.maximum(near, 0)], 0.0).max(1))
    c_u = 2.0 * N * CM * np.abs(np.asarray(s.H)).max() + rates + 4.0 * link
    bar = 2.0 ** -53 * (4 * N + 20) * c_u * m_u * scale + 200 * 5e-324
    ref = ore * scale + 1j * (oim * scale)
    assert np.all(np.abs(gre[us] + 1j * gim[us] - ref) <= bar[:, None, None])


@pytest.mark.parametrize("N,D,herm,cplx,general", CASES)
@pytest.mark.parametrize("scale", [1.0, 1e-150, 1e-285, 1e-320, 1e285])
def test_every_ado_to_its_own_scale(heom, N, D, herm, cplx, general, scale):
    _check(heom, N, D, herm, cplx, general, scale)


@pytest.mark.parametrize("N,D", COLUMN)
def test_column_kernel_every_ado_to_its_own_scale(heom, N, D):
    _check(heom, N, D, True, False, False, 1.0)


@pytest.mark.parametrize("N,D", [(8, 8), (16, 4)])
@pytest.mark.parametrize("scale", [1e-150, 1e-285, 1e-320, 1e285])
def test_column_kernel_at_the_ends_of_the_range(heom, N, D, scale):
    _check(heom, N, D, True, False, False, scale)


@pytest.mark.parametrize("N,D", COLUMN)
def test_column_kernel_steps(heom, N, D):
    """Two steps from a site, sampled ADOs within 1e-12 of the oracle; the run takes four launches a step, not one for many:
    the column kernel."""
    s = _system(N, D)
    rho = np.zeros((N, N))
    rho[0, 0] = 1.0
    m, ore, oim, oobs = oracle_propagate(wl.Propagation(s, rho, np.zeros((N, N)), 0.5, 2), 2, stride=1)
    r = _run(heom, s)
    before = r.launches()
    r.propagate(0.5, 2, 1)
    assert r.launches() - before >= 8
    re, im = r.get_ados(0, r.n_ado)
    assert np.max(np.abs(re + 1j * im - (ore + 1j * oim))) <= 1e-12
    assert np.max(np.abs(r.observables()[:, :N + 4] - oobs)) <= 1e-12
    r.close()


@pytest.mark.parametrize("N,D", [(8, 8), (13, 6), (16, 4)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_column_kernel_non_finite_stays_visible(heom, N, D, bad):
    """An Inf or NaN in one ADO makes that ADO's right-hand side non-finite and leaves ADOs without a link to it finite."""
    s = _system(N, D)
    r = _run(heom, s)
    rng = np.random.default_rng(3)
    x = rng.standard_normal((r.n_ado, N, N))
    x = 0.5 * (x + np.transpose(x, (0, 2, 1)))
    x[0, 2, 2] = bad
    r.set_ados(0, x, np.zeros_like(x))
    gre, gim = r.rhs_eval(0, r.n_ado)
    r.close()
    level2 = 1 + N
    assert not np.all(np.isfinite(gim[0]))
    assert np.all(np.isfinite(gre[level2:])) and np.all(np.isfinite(gim[level2:]))
