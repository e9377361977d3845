"""Rounds that rebuild the messages from the nodes' last aggregates, against
the FP64 oracle: sizes around the tile edge, the rounds in which the kernels
change (first, live P, frozen P with fewer and fewer terms, a restart), data on
both sides of the line where messages are stored instead, every form of Q.

Bars: relative mean error 2e-5 as for every round (Q entries to 1e-6, FP32
aggregates, a contracting round; what a round leaves out is at most 2^-24 of the
largest mean), messages to 1e-4 relative plus 1e-6 of the largest, as stored
messages are held to.
"""
import numpy as np
import pytest

import oracle
from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu

REL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


def _problem(n, m, g, near):
    """A mixture with width g / m; `near` pairs of near-duplicates that a narrow
    kernel leaves with few other neighbours."""
    p = workloads.mixture(n, m, seed=7 * n + m, gamma=g / m, C=10.0)
    X = p.X.copy()
    for k in range(near):
        X[2 * k + 1] = X[2 * k] + 1e-2
    return workloads.Problem(X, p.y, p.gamma, p.C)


# wide kernels (few orders), narrow ones (all orders), and strongly coupled
# pairs (stored messages)
CASES = [(127, 6, 0.2, 0), (128, 6, 0.5, 0), (129, 20, 1.0, 0), (257, 8, 1.0, 0), (640, 8, 2.0, 0), (384, 32, 2.0, 4),
         (200, 64, 8.0, 3)]


@pytest.mark.parametrize("n,m,g,near", CASES)
@pytest.mark.parametrize("stages", [1, 3])
def test_rounds_match_oracle(n, m, g, near, stages):
    p = _problem(n, m, g, near)
    Q = oracle.build_q(p.X.astype(np.float64), p.y.astype(np.float64), p.gamma, p.C)
    s = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, stages=stages)
    rng = np.random.default_rng(n)
    i = rng.integers(0, n - 1, 200)
    j = rng.integers(i + 1, n)
    for iters in (1, 2, 3, 4, 6, 9, 30):
        s.refit(p.X, p.y, p.gamma, p.C)
        s.solve(iters, 0.0)
        r = (oracle.gabp(Q, np.ones(n), iters=iters, keep_messages=True) if stages == 1
             else oracle.gabp_staged(Q, np.ones(n), iters=iters, stages=stages, block=128))
        assert np.max(np.abs(s.mean() - r.mu)) <= REL * np.max(np.abs(r.mu)), iters
        if stages == 1:
            got = gabp.svm_get_pairs(s.h, i, j).astype(np.float64)
            want = np.stack([r.Pin[j, i], r.Pin[i, j], r.Hin[j, i], r.Hin[i, j]], axis=1)
            np.testing.assert_allclose(got, want, rtol=1e-4, atol=1e-6 * np.max(np.abs(want)))


@pytest.mark.parametrize("n,m,g,near", [(300, 8, 0.5, 0), (200, 64, 8.0, 3)])
@pytest.mark.parametrize("stages", [1, 4])
def test_resumed_solve_equals_one_call(n, m, g, near, stages):
    """The final pass of a solve leaves the sums alone that the next round
    reads (staged rounds read those of tiles not swept yet)."""
    p = _problem(n, m, g, near)
    s = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, stages=stages)
    for k in (1, 2, 3, 6):
        s.solve(k, 0.0)
    one = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, stages=stages).solve(12, 0.0)[0]
    np.testing.assert_array_equal(s.solve(0, 0.0)[0], one)


@pytest.mark.parametrize("kw", [dict(q_mode=gabp.Q_BF16), dict(q_mode=gabp.Q_RECOMPUTE),
                                dict(q_mode=gabp.Q_RECOMPUTE, msg_bf16=1, stages=2), dict(task=gabp.TASK_KRR)])
@pytest.mark.parametrize("n,m,g", [(129, 70, 0.5), (385, 8, 2.0)])
def test_forms_reach_the_solve(kw, n, m, g):
    """Refined BF16 forms (their restarts of H included) and the regression task
    to tolerance, on the linear solve."""
    p = _problem(n, m, g, 0)
    X = p.X.astype(np.float64)
    if "q_mode" in kw:
        kw = dict(kw, refine=10)
    if kw.get("task"):
        t = workloads.krr_targets(p, 3)
        Q, b, C = oracle.build_q_krr(X, p.gamma, 0.5), t.astype(np.float64), 0.5
        s = gabp.GabpSVM(p.X, t, p.gamma, C, **kw)
    else:
        Q, b = oracle.build_q(X, p.y.astype(np.float64), p.gamma, p.C), np.ones(n)
        s = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, **kw)
    s.solve(300, 1e-6)
    assert s.stats()["converged"] == 1
    ref = np.linalg.solve(Q, b)
    assert np.max(np.abs(s.mean() - ref)) <= REL * np.max(np.abs(ref))


@pytest.mark.parametrize("n,g", [(900, 2.0), (1410, 0.5), (1665, 0.1)])
@pytest.mark.parametrize("stages", [1, 3])
def test_rounds_of_fewer_orders_match_oracle(n, g, stages):
    """Larger sets, whose live rounds sum fewer and fewer orders (q^2 to q^4 with
    q^3, q^2 and q^3, q^2 alone), on both schedules."""
    p = _problem(n, 8, g, 0)
    Q = oracle.build_q(p.X.astype(np.float64), p.y.astype(np.float64), p.gamma, p.C)
    s = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, stages=stages)
    for iters in (1, 2, 3, 5, 12):
        s.refit(p.X, p.y, p.gamma, p.C)
        s.solve(iters, 0.0)
        r = (oracle.gabp(Q, np.ones(n), iters=iters) if stages == 1
             else oracle.gabp_staged(Q, np.ones(n), iters=iters, stages=stages, block=128))
        assert np.max(np.abs(s.mean() - r.mu)) <= REL * np.max(np.abs(r.mu)), iters
