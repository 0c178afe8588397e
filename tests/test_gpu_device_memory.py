"""Device memory that the runtime takes by itself: the local memory of a kernel (its stack times every thread that the
GPU can hold) stays with the context from the first launch on.  heom_propagate_static is for callers that own all
device memory, so the small runs that it takes must not cost any to speak of.  In a fresh process, after a first FP64 call
(context, library, static workspace), calls of every form of whole-step launch together leave the free memory as it was but
for their code: 64 MiB allowed; a stack of 2.6 KB a thread took 468 MiB."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))

CODE = """
import numpy as np
import torch
from paper_1803_03498_gb300 import heom
from paper_1803_03498_gb300 import workloads as wl


def call(N, K, D, precision, start):
    rng = np.random.default_rng(N)
    H = np.diag(rng.uniform(0.0, 400.0, N)) + np.triu(rng.normal(0.0, 40.0, (N, N)), 1)
    H = H + np.triu(H, 1).T
    s = wl.System("s", H, list(range(N)), [35.0] * N, [60.0] * N, [300.0] * N, K=K, D=D)
    re = np.zeros((N, N))
    re[0, 0] = 1.0
    re[-1, 0] = start
    heom.propagate_static(s, re, precision=precision, dt_fs=0.5, n_steps=8, obs_stride=4)


call(2, 0, 4, "fp64", 0.0)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for N, K, D, precision, start in [(2, 0, 4, "fp32_mixed", 0.0), (7, 1, 3, "fp32_mixed", 0.0), (22, 0, 2, "fp32_mixed", 0.0),
                                  (24, 0, 2, "fp32_mixed", 0.0), (7, 1, 3, "fp32_mixed", 0.5), (7, 1, 3, "fp64", 0.5),
                                  (14, 0, 2, "fp64", 0.0), (23, 0, 2, "fp64", 0.0)]:
    call(N, K, D, precision, start)
torch.cuda.synchronize()
print("fell by", free - torch.cuda.mem_get_info()[0])
"""


def test_whole_step_launches_take_no_device_memory():
    from paper_1803_03498_gb300.build import build
    build()
    p = subprocess.run([sys.executable, "-c", CODE], cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    assert int(p.stdout.split("fell by")[1]) <= 64 << 20, p.stdout
