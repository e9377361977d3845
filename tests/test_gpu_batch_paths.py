"""Batches and servers that hold both kinds of instances, those that keep a history
of their nodes and those that store their messages (near-duplicate points that a
narrow kernel leaves with few other neighbours): each member's result is the one
it has alone, bit for bit, also where a slot goes from one kind to the other.
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


def _problem(n, stored):
    if not stored:
        return workloads.mixture(n, 8, seed=n, gamma=0.5 / 8, C=10.0)
    p = workloads.mixture(n, 64, seed=n, gamma=8.0 / 64, C=10.0)
    X = p.X.copy()
    X[1] = X[0] + 1e-2
    X[n // 2] = X[n - 1] + 1e-2
    return workloads.Problem(X, p.y, p.gamma, p.C)


SIZES = [(300, False), (200, True), (513, True), (640, False), (129, True), (900, False)]
FORMS = [{}, {"stages": 3}, {"q_mode": gabp.Q_BF16, "refine": 6}, {"q_mode": gabp.Q_BF16, "refine": 6, "msg_bf16": 1, "stages": 2},
         {"q_mode": gabp.Q_RECOMPUTE, "refine": 6}]


def test_the_problems_are_of_both_kinds():
    """Strongest coupling |q| / d at the start: the line lies at 1/4."""
    for n, stored in SIZES:
        p = _problem(n, stored)
        Q = oracle.build_q(p.X.astype(np.float64), p.y.astype(np.float64), p.gamma, p.C)
        u = np.abs(Q - np.diag(np.diag(Q))).max() / np.diag(Q).min()
        pair = np.max(np.abs(Q - np.diag(np.diag(Q))) / np.diag(Q)[:, None])
        assert pair > 0.5 if stored else u < 0.1, (n, u, pair)


def _alone(p, iters, tol, kw):
    svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, chunk=4, **kw)
    alpha = np.array(svm.solve(iters, tol)[0])
    out = alpha, np.array(svm.mean()), svm.stats()["converged"]
    svm.close()
    return out


@pytest.mark.parametrize("kw", FORMS)
@pytest.mark.parametrize("iters,tol", [(9, 0.0), (300, 1e-6)])
def test_batch_equals_alone(kw, iters, tol):
    ps = [_problem(n, stored) for n, stored in SIZES]
    alphas, res, _ = gabp.batch_solve(ps, iters, tol, means=True, chunk=4, **kw)
    for p, a, r in zip(ps, alphas, res):
        alpha, mu, converged = _alone(p, iters, tol, kw)
        assert r["status"] == 0 and r["converged"] == converged
        np.testing.assert_array_equal(a, alpha)
        np.testing.assert_array_equal(r["mu"], mu)


@pytest.mark.parametrize("kw", FORMS)
def test_server_slots_go_from_one_kind_to_the_other(kw):
    ps = [_problem(n, stored) for n, stored in SIZES * 2]
    srv = gabp.Server(iters=300, tol=1e-6, max_members=2, chunk=4, **kw)
    tickets = [srv.submit(p.X, p.y, p.gamma, p.C) for p in ps]
    out = {}
    for _ in range(4000):
        srv.step()
        for t in srv.completed():
            out[t] = srv.poll(t)
        if len(out) == len(ps):
            break
    srv.close()
    assert len(out) == len(ps)
    for p, t in zip(ps, tickets):
        a, r = out[t]
        alpha, _, converged = _alone(p, 300, 1e-6, kw)   # (n = 129 stops at an FP32 floor of 3e-6)
        assert r["status"] == 0 and r["converged"] == converged
        np.testing.assert_array_equal(a, alpha)
