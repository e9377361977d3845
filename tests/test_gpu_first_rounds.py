"""The first rounds of instances that store no messages, where the terms that later
rounds have are still missing: every round count up to 6, in one solve and resumed,
before and after a restart of the H messages, against FP64 GaBP written out on the
dense matrix that the handle holds.

Bar: 2e-6 of the largest mean up to that round.  A mean is a sum of products q mu
of FP32 entries, which the matrix read back carries exactly: what is left is the
rounding of the sums, a few units of 2^-24 of sum |q mu| / Q_ii <= max |mu| a round
(32 of them: 1.9e-6; measured, 1e-7).
"""
import numpy as np
import pytest

from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu

BAR = 2e-6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


def _problem(n, m, g, same):
    p = workloads.mixture(n, m, seed=n + m, gamma=g / m, C=10.0)
    X = p.X.copy()
    if same:
        X[:] = X[0] + 1e-3 * X
    return workloads.Problem(X, p.y, p.gamma, p.C)


class Dense:
    """Algorithm 2 and its staged schedule on a dense matrix, in FP64."""

    def __init__(self, Q, b, stages):
        n = len(b)
        self.d, self.b = np.diag(Q).copy(), b
        self.q = Q - np.diag(self.d)
        self.P, self.H = np.zeros((n, n)), np.zeros((n, n))   # [i, j]: the message i -> j
        nt = (n + 127) // 128
        edge = [0] * (stages + 1)
        for k in range(1, stages):
            e = edge[k - 1]
            while e < nt and stages * (e * (e + 1) // 2) < k * (nt * (nt + 1) // 2):
                e += 1
            edge[k] = e
        edge[stages] = nt
        band = np.maximum.outer(np.arange(n) // 128, np.arange(n) // 128)
        self.masks = [(band >= edge[k]) & (band < edge[k + 1]) for k in range(stages)]

    def round(self):
        for m in self.masks:
            Pt, ht = self.d + self.P.sum(0), self.b + self.H.sum(0)
            den = Pt[:, None] - self.P.T
            P, H = -self.q ** 2 / den, -self.q * (ht[:, None] - self.H.T) / den
            self.P, self.H = np.where(m, P, self.P), np.where(m, H, self.H)

    def mean(self):
        return (self.b + self.H.sum(0)) / (self.d + self.P.sum(0))


# all entries near 1 (the largest z of this path that so few points can have), an
# ordinary kernel, and sizes of several tiles
CASES = [(30, 3, 0.5, True), (33, 64, 0.5, True), (129, 8, 0.2, False), (300, 8, 1.0, False), (520, 8, 0.5, True)]


@pytest.mark.parametrize("n,m,g,same", CASES)
@pytest.mark.parametrize("stages", [1, 3])
@pytest.mark.parametrize("task", [0, 1])
@pytest.mark.parametrize("q_mode", [gabp.Q_F32, gabp.Q_BF16])
def test_first_rounds(n, m, g, same, stages, task, q_mode):
    p = _problem(n, m, g, same)
    y = workloads.krr_targets(p, 4) if task else p.y
    for split in (False, True):
        svm = gabp.GabpSVM(p.X, y, p.gamma, p.C, stages=stages, task=task, q_mode=q_mode)
        Q = gabp.svm_get_q(svm.h, n).astype(np.float64)
        ref = Dense(Q, y.astype(np.float64) if task else np.ones(n), stages)
        largest = np.abs(ref.mean()).max()
        for k in range(1, 7):
            ref.round()
            largest = max(largest, np.abs(ref.mean()).max())
            if split:
                svm.solve(1, 0.0)
            else:
                svm.refit(p.X, y, p.gamma, p.C)
                svm.solve(k, 0.0)
            assert np.abs(svm.mean() - ref.mean()).max() <= BAR * largest, (k, split)
        svm.close()


@pytest.mark.parametrize("n,m,g,same", CASES)
@pytest.mark.parametrize("stages", [1, 3])
@pytest.mark.parametrize("iters", [1, 2, 3])
def test_first_rounds_after_a_restart(n, m, g, same, stages, iters):
    """One correction pass of `iters` rounds: the H messages restart, the P messages
    go on."""
    p = _problem(n, m, g, same)
    kw = dict(stages=stages, q_mode=gabp.Q_BF16, refine_handover=1e-30, refine_inner=1e-30)
    got = {}
    for refine in (0, 1):
        svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, refine=refine, **kw)
        Q = gabp.svm_get_q(svm.h, n).astype(np.float64)
        svm.solve(iters, 0.0)
        got[refine] = svm.mean().astype(np.float64)
        svm.close()
    exact = gabp.GabpSVM(p.X, p.y, p.gamma, p.C)
    Q32 = gabp.svm_get_q(exact.h, n).astype(np.float64)
    exact.close()
    ref = Dense(Q, np.ones(n), stages)
    for _ in range(iters):
        ref.round()
    r = np.ones(n) - Q32 @ got[0]       # the residual of the handle's own first solve
    ref.b, ref.H = r, np.zeros((n, n))
    largest = np.abs(ref.mean()).max()
    for _ in range(iters):
        ref.round()
        largest = max(largest, np.abs(ref.mean()).max())
    # the correction, and the rounding of the sum of both
    bar = BAR * largest + 2.0 ** -23 * np.abs(got[1]).max()
    assert np.abs((got[1] - got[0]) - ref.mean()).max() <= bar
