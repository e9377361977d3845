"""A batch does not run more rounds than its limit: with a limit of one round, long
chunks take the call no longer than chunks of one, and the results are those of
the limit.

Bar: a factor of 1.3 (63 rounds for nothing doubled the call and more).
"""
import time

import numpy as np
import pytest

from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


@pytest.mark.parametrize("kw", [{}, {"stages": 3}, {"q_mode": gabp.Q_RECOMPUTE, "refine": 4}])
def test_short_limits_stay_short(kw):
    ps = [workloads.mixture(n, 8, seed=n) for n in (200, 700, 1300, 3000)]

    def best(chunk):
        out = []
        for _ in range(8):
            t = time.perf_counter()
            gabp.batch_solve(ps, 1, 0.0, chunk=chunk, **kw)
            out.append(time.perf_counter() - t)
        return min(out[1:])

    assert best(64) <= 1.3 * best(1)


@pytest.mark.parametrize("kw", [{}, {"stages": 3}, {"q_mode": gabp.Q_RECOMPUTE, "refine": 4}])
@pytest.mark.parametrize("chunk", [0, 64])
@pytest.mark.parametrize("iters", [1, 3])
def test_short_limits_equal_alone(kw, chunk, iters):
    ps = [workloads.mixture(n, 8, seed=n) for n in (200, 700, 1300)]
    alphas, res, _ = gabp.batch_solve(ps, iters, 0.0, chunk=chunk, **kw)
    for p, a, r in zip(ps, alphas, res):
        svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, **kw)
        np.testing.assert_array_equal(a, np.array(svm.solve(iters, 0.0)[0]))
        svm.close()
        if not kw.get("refine"):
            assert r["iters_done"] == iters
