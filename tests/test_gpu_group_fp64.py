"""Small FP64 runs share launches of whole steps in heom_group_propagate: several runs in one grid, each with CTAs and a
barrier of its own.  Every run must come out as it does alone, bit for bit: more runs than one launch holds, more CTAs than
keep their ADOs at once, runs whose steps end inside and between launches, that start at different steps and record
every few steps, of every kind (with and without fixed point, two sizes of pairs, element form, not Hermitian, complex H),
beside mixed and column-0 runs in the same call."""
import numpy as np
import pytest

from paper_1803_03498_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def heom():
    from paper_1803_03498_gb300.build import build
    build()
    from paper_1803_03498_gb300 import heom as h
    h.load()
    return h


def _prop(N, K, D, seed, start="site", cplx=False):
    rng = np.random.default_rng(1803600 + seed)
    H = np.diag(rng.uniform(0.0, 400.0, N)) + np.triu(rng.normal(0.0, 40.0, (N, N)), 1)
    H = H + np.triu(H, 1).T
    if cplx:
        A = np.triu(rng.normal(0.0, 20.0, (N, N)), 1)
        H = H + 1j * (A - A.T)
    s = wl.System(f"N={N}", H, list(range(N)), list(rng.uniform(20, 100, N)), [60.0] * N, [300.0] * N, K=K, D=D)
    re, im = np.zeros((N, N)), np.zeros((N, N))
    if start == "site":
        re[0, 0] = 1.0
    else:
        re[:, 0], im[:, 0] = rng.normal(size=N), rng.normal(size=N)
    return wl.Propagation(s, re, im, 0.5, 0)


def _compare(heom, cases, steps, before, stride, sample=None):
    """cases: (propagation, precision); each run takes before[i] steps alone, then steps[i] with the others."""
    def run(i):
        p, precision = cases[i]
        r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision=precision, w=p.w,
                     max_records=(steps[i] + before[i]) // stride + 1)
        r.propagate(0.5, before[i], stride)
        return r

    runs = [run(i) for i in range(len(cases))]
    launches = [r.launches() for r in runs]
    heom.group_propagate(runs, 0.5, steps, obs_stride=stride)
    for i in (range(len(cases)) if sample is None else sample):
        r, one = runs[i], run(i)
        one.propagate(0.5, steps[i], stride)
        assert r.info() == one.info()
        if cases[i][1] == "fp64":  # whole steps: far fewer launches than four a step
            assert r.launches() - launches[i] <= 1 + steps[i], cases[i][0].system.name
        assert np.array_equal(r.observables(), one.observables()), cases[i][0].system.name
        a, b = r.get_ados(0, r.n_ado), one.get_ados(0, r.n_ado)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), cases[i][0].system.name
        one.close()
    for r in runs:
        r.close()


def test_more_small_runs_than_one_launch_holds(heom):
    """300 runs of 2 to 4 states, 1 to 150 steps (launches take up to 64), three of them at other starts."""
    rng = np.random.default_rng(1)
    cases = [(_prop(2 + i % 3, 0, 2 + i % 2, i), "fp64") for i in range(300)]
    steps = [int(x) for x in rng.integers(1, 151, 300)]
    steps[0], steps[1], steps[2], steps[299] = 64, 65, 128, 150
    before = [0] * 300
    before[3], before[100], before[298] = 5, 7, 66
    _compare(heom, cases, steps, before, 4, [0, 1, 2, 3, 4, 100, 150, 254, 255, 256, 257, 298, 299])


def test_more_ctas_than_can_keep_their_ados(heom):
    """12 runs of 3060 ADOs of 7 x 7 (279 CTAs each to be kept) and one of 120: all in chunks."""
    cases = [(_prop(7, 1, 4, i), "fp64") for i in range(12)] + [(_prop(7, 0, 3, 50), "fp64")]
    _compare(heom, cases, [3 + i for i in range(12)] + [20], [0] * 12 + [3], 3, [0, 1, 5, 11, 12])


def test_every_kind_in_one_call(heom):
    cases = [(_prop(1, 1, 2, 1), "fp64"), (_prop(3, 0, 4, 2), "fp64"), (_prop(7, 1, 3, 3), "fp64"),
             (_prop(7, 1, 4, 4), "fp64"), (_prop(9, 0, 3, 5), "fp64"), (_prop(14, 1, 2, 6), "fp64"),
             (_prop(22, 0, 2, 7), "fp64"), (_prop(23, 0, 2, 8), "fp64"), (_prop(24, 0, 1, 9), "fp64"),
             (_prop(7, 1, 2, 10, "coherence"), "fp64"), (_prop(18, 0, 2, 11, "coherence"), "fp64"),
             (_prop(6, 1, 2, 12, cplx=True), "fp64"), (_prop(12, 0, 2, 13, "coherence", True), "fp64"),
             (_prop(7, 1, 3, 14), "fp32_mixed"), (_prop(5, 0, 3, 15, "coherence"), "fp32_mixed"),
             (_prop(19, 0, 2, 16), "fp32_mixed")]
    rng = np.random.default_rng(2)
    steps = [int(x) for x in rng.integers(1, 90, len(cases))]
    steps[1] = 0
    runs_before = [int(x) for x in rng.integers(0, 6, len(cases))]
    _compare(heom, cases, steps, runs_before, 5)


def test_mixed_and_column_runs_beside_small_fp64_runs(heom):
    dip = wl.fmo_like()[1][1]
    cases = [(_prop(7, 1, 4, 4), "fp64"), (_prop(7, 1, 3, 14), "fp32_mixed"), (_prop(12, 0, 3, 20), "fp32_mixed"),
             (dip, "fp32_mixed"), (_prop(9, 0, 3, 5), "fp64")]
    _compare(heom, cases, [40, 37, 20, 33, 70], [0, 2, 0, 1, 3], 3)
