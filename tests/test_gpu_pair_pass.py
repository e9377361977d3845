"""The pass over the pairs that decides how an instance holds its messages, where
many tiles settle the question at once: its outcome does not depend on which warp
finds a strongly coupled pair first, so the same data give the same bits.

Bar of the means: 2e-5 of the largest, as every round is held to against FP64.
"""
import numpy as np
import pytest

import oracle
from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


def _problem(n, near):
    """A narrow kernel, with `near` near-duplicate pairs spread over the tiles."""
    p = workloads.mixture(n, 64, seed=n + near, gamma=8.0 / 64, C=10.0)
    X = p.X.copy()
    for k in range(near):
        a, b = (37 * k) % (n // 2), n // 2 + (53 * k) % (n // 2)
        X[b] = X[a] + 1e-2
    return workloads.Problem(X, p.y, p.gamma, p.C)


@pytest.mark.parametrize("n,near", [(1500, 0), (1500, 1), (1500, 200), (2049, 1000)])
@pytest.mark.parametrize("kw", [{}, {"q_mode": gabp.Q_BF16, "refine": 3}, {"q_mode": gabp.Q_RECOMPUTE, "refine": 3}])
def test_choice_is_repeatable(n, near, kw):
    p = _problem(n, near)
    svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, **kw)
    first = None
    for _ in range(12):
        svm.refit(p.X, p.y, p.gamma, p.C)
        svm.solve(12, 0.0)
        mu = np.array(svm.mean())
        first = mu if first is None else first
        assert np.array_equal(mu, first)
    svm.close()
    if not kw:
        Q = oracle.build_q(p.X.astype(np.float64), p.y.astype(np.float64), p.gamma, p.C)
        ref = oracle.gabp(Q, np.ones(n), iters=12).mu
        assert np.max(np.abs(first - ref)) <= 2e-5 * np.max(np.abs(ref))


def test_batch_of_both_kinds_is_repeatable():
    ps = [_problem(n, near) for n, near in ((700, 0), (900, 300), (513, 1), (1200, 600))]
    first = None
    for _ in range(8):
        _, res, _ = gabp.batch_solve(ps, 12, 0.0, means=True)
        mu = [np.array(r["mu"]) for r in res]
        first = mu if first is None else first
        assert all(np.array_equal(a, b) for a, b in zip(mu, first))
