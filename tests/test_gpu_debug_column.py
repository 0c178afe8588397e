"""The bounds-checked debug build (see test_gpu_debug_build.py) on the kernels that its small cases do not reach: the column
kernel, whose hierarchies lie above those of whole-step launches, and launches of whole steps with several runs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))

CODE = """
import sys
sys.path.insert(0, {here!r})
import numpy as np
from helpers import oracle_propagate
from paper_1803_03498_gb300 import heom
from paper_1803_03498_gb300 import workloads as wl

print("library", heom.LIB_PATH)


def prop(N, K, D):
    rng = np.random.default_rng(N)
    H = np.diag(rng.uniform(0.0, 400.0, N)) + np.triu(rng.normal(0.0, 40.0, (N, N)), 1)
    s = wl.System("s", H + np.triu(H, 1).T, list(range(N)), [35.0] * N, [60.0] * N, [300.0] * N, K=K, D=D)
    rho = np.zeros((N, N))
    rho[0, 0] = 1.0
    return wl.Propagation(s, rho, np.zeros((N, N)), 0.5, 2)


for N, D in [(8, 8), (12, 6), (16, 4)]:
    p = prop(N, 0, D)
    m, ore, oim, oobs = oracle_propagate(p, 2, stride=1)
    r = heom.Run(p.system, p.rho0_re, p.rho0_im, precision="fp64", max_records=4)
    before = r.launches()
    r.propagate(0.5, 2, 1)
    assert r.launches() - before >= 8  # stage launches: the column kernel
    assert np.max(np.abs(r.observables()[:, :N + 4] - oobs)) <= 1e-12
    re, im = r.get_ados(0, r.n_ado)
    assert np.max(np.abs(re + 1j * im - (ore + 1j * oim))) <= 1e-12
    r.close()
ps = [prop(N, 0, 3) for N in (2, 5, 7, 9, 14, 18, 22, 23)]
runs = [heom.Run(p.system, p.rho0_re, p.rho0_im, precision="fp64", max_records=4) for p in ps]
heom.group_propagate(runs, 0.5, 20, obs_stride=10)
for p, r in zip(ps, runs):
    m, ore, oim, oobs = oracle_propagate(p, 20, stride=10)
    assert np.max(np.abs(r.observables()[:, :p.system.N + 4] - oobs)) <= 1e-12
print("ALL OK")
"""


def test_debug_build_column_kernel_and_shared_launches():
    from paper_1803_03498_gb300.build import build
    lib = build(debug=True)
    p = subprocess.run([sys.executable, "-c", CODE.format(here=HERE)], cwd=os.path.dirname(HERE), capture_output=True,
                       env=dict(os.environ, HEOM_LIB=lib), text=True, timeout=900)
    out = p.stdout + p.stderr
    assert p.returncode == 0, out[-3000:]
    assert f"library {lib}" in out and "ALL OK" in out
