"""FP64 runs hold FP64: every element of a right-hand side is as precise as a chain of FP64 multiply-adds over its own
terms, however small it is beside the others of its ADO.

The state is non-zero on one level of the hierarchy only.  Links join neighbouring levels, so on that level the
right-hand side is -i [H, z] - (g_u + T) z, which is computed here in extended precision.  The bar is the rounding bound of
such a chain, element by element: (2 N + 8) units of 2^-53 of the sum of the terms' magnitudes (2 N products, the decay,
H in rad/fs, the rates); a commutator that keeps only the leading bits of its operands' largest element misses it
by many orders of magnitude on weak elements."""
import numpy as np
import pytest

from paper_1803_03498_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

LD = np.longdouble
CM = 2.0 * np.pi * 2.99792458e-5  # rad/fs per cm^-1


@pytest.fixture(scope="module")
def heom():
    from paper_1803_03498_gb300.build import build
    build()
    from paper_1803_03498_gb300 import heom as h
    h.load()
    return h


def _system(N, K, D, cplx=False):
    """Site energies 0..400 cm^-1, couplings of 40 cm^-1, those of the last state 1e-6 cm^-1."""
    rng = np.random.default_rng(1803500 + N)
    H = np.diag(np.round(rng.uniform(0.0, 400.0, N))) + np.triu(rng.normal(0.0, 40.0, (N, N)), 1)
    H[:-1, -1] *= 2.5e-8
    H = H + np.triu(H, 1).T
    if cplx:
        A = np.triu(rng.normal(0.0, 20.0, (N, N)), 1)
        H = H + 1j * (A - A.T)
    return wl.System(f"N={N}", H, list(range(N)), [35.0] * N, [60.0] * N, [300.0] * N, K=K, D=D)


def _tiles(rng, count, N, kind, herm):
    """Tiles with weak elements beside strong ones: |psi><psi| of states over five decades, elements over twelve
    decades each, or one strong element beside weak ones."""
    z = rng.standard_normal((count, N, N)) + 1j * rng.standard_normal((count, N, N))
    if kind == "pure":
        w = 10.0 ** -rng.uniform(0.0, 5.0, (count, N))
        z *= w[:, :, None] * w[:, None, :]
    elif kind == "spread":
        z = z * 10.0 ** -rng.uniform(0.0, 12.0, (count, N, N))
    else:
        z *= 1e-9
        z[:, 0, 0] = 1.0
    return 0.5 * (z + np.conj(np.transpose(z, (0, 2, 1)))) if herm else z


# (states, K, depth, precision, level, Hermitian, complex H, general): the pair kernels with and without fixed point,
# the element kernels, the FP64 head of a mixed run and the column kernel
CASES = [(7, 1, 4, "fp64", 3, True, False, False), (7, 1, 2, "fp64", 1, True, False, False),
         (9, 0, 3, "fp64", 2, True, False, False), (16, 0, 3, "fp64", 3, True, False, False),
         (22, 0, 2, "fp64", 2, True, False, False), (23, 0, 2, "fp64", 2, True, False, False),
         (18, 0, 2, "fp64", 2, False, False, False), (6, 1, 2, "fp64", 1, True, True, False),
         (12, 0, 2, "fp64", 2, False, True, False), (9, 0, 2, "fp64", 2, True, False, True),
         (14, 1, 2, "fp32_mixed", 1, True, False, False), (23, 0, 2, "fp32_mixed", 1, True, False, False),
         (8, 0, 10, "fp64", 9, True, False, False), (14, 1, 4, "fp64", 4, True, False, False),
         (16, 0, 5, "fp64", 5, True, False, False)]


@pytest.mark.parametrize("N,K,D,precision,level,herm,cplx,general", CASES)
@pytest.mark.parametrize("kind", ["pure", "spread", "one"])
def test_weak_elements_keep_fp64_precision(heom, N, K, D, precision, level, herm, cplx, general, kind):
    s = _system(N, K, D, cplx)
    rho = np.zeros((N, N))
    rho[0, 0] = 1.0
    r = heom.Run(s, rho, np.zeros((N, N)), precision=precision, max_records=2, time_dependent=general)
    lo, hi = int(r.hier.level_offsets[level]), int(r.hier.level_offsets[level + 1])
    rng = np.random.default_rng(N)
    z = np.zeros((r.n_ado, N, N), dtype=complex)
    z[lo:hi] = _tiles(rng, hi - lo, N, kind, herm)
    r.set_ados(0, z.real, z.imag)
    gre, gim = r.rhs_eval(0, r.n_ado)
    n, _, _ = r.hier.export()
    r.close()
    modes = heom.bath_modes(s)
    T = modes["term"][:, None] + modes["term"][None, :]
    T[np.diag_indices(N)] = 0.0
    H = np.asarray(s.H)
    d = H.diagonal().real
    Hr = CM * (H.real - np.eye(N) * 0.5 * (d.max() + d.min()))
    Hi = CM * H.imag
    us = np.unique(np.concatenate([[lo, lo + 1, hi - 1], rng.integers(lo, hi, 150)]))
    zr, zi = z[us].real.astype(LD), z[us].imag.astype(LD)
    hr, hi_ = Hr.astype(LD), Hi.astype(LD)
    f = (n[us].astype(float) @ modes["gamma"])[:, None, None] + T
    br = (hr @ zr - hi_ @ zi) - (zr @ hr - zi @ hi_)  # [H, z]
    bi = (hr @ zi + hi_ @ zr) - (zr @ hi_ + zi @ hr)
    ar, ai, yr, yi = abs(hr), abs(hi_), abs(zr), abs(zi)
    tr = (ar @ yr + ai @ yi) + (yr @ ar + yi @ ai)
    ti = (ar @ yi + ai @ yr) + (yr @ ai + yi @ ar)
    units = (2 * N * (2 if cplx else 1) + 8) * 2.0 ** -53
    assert np.all(np.abs(gre[us] - (bi - f * zr)) <= units * (ti + f * yr))
    assert np.all(np.abs(gim[us] - (-br - f * zi)) <= units * (tr + f * yi))
