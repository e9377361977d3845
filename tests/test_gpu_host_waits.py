"""A program that has asked CUDA's waits to block gets its core back while a solve
runs, and the same bits as one that lets them spin.

Bar: a solve of 0.2 s takes its thread less than half of that (launches and
captures take a few per cent, a wait that polls takes all of it).
"""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, hashlib, sys, time
flags, stages, tol = int(sys.argv[1]), int(sys.argv[2]), float(sys.argv[3])
cu = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
if flags:
    assert cu.cuDevicePrimaryCtxSetFlags_v2(dev, flags) == 0
import numpy as np
from paper_0810_1648_gb300 import gabp, workloads
p = workloads.mixture(20000, 16, seed=3)
svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, stages=stages)
svm.solve(2, 0.0)
svm.refit(p.X, p.y, p.gamma, p.C)
w, c = time.perf_counter(), time.thread_time()
alpha = svm.solve(1500, tol)[0]
w, c = time.perf_counter() - w, time.thread_time() - c
print(w, c, hashlib.sha256(np.array(alpha).tobytes()).hexdigest())
"""
SPIN, YIELD, BLOCK = 1, 2, 4


def _run(flags, stages, tol):
    out = subprocess.run([sys.executable, "-c", CHILD, str(flags), str(stages), str(tol)], capture_output=True, text=True,
                         timeout=120)
    assert out.returncode == 0, out.stderr[-2000:]
    w, c, digest = out.stdout.split()
    return float(w), float(c), digest


@pytest.mark.parametrize("stages", [1, 4])
@pytest.mark.parametrize("tol", [0.0, 1e-30])
def test_blocking_waits_are_honoured(stages, tol):
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()
    wall, cpu, bits = _run(BLOCK, stages, tol)
    assert wall > 0.1
    assert cpu < 0.5 * wall, (cpu, wall)
    assert bits == _run(0, stages, tol)[2] == _run(YIELD, stages, tol)[2]
