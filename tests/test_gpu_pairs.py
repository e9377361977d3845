"""Messages read back from a handle that recomputes Q are those of the handle that
stores the same BF16 entries, bit for bit: both hold the same rounds, and a pair's
messages are rebuilt from the entry that the rounds used.  Exact, like the rounds
themselves (test_recompute_equals_bf16_store).
"""
import numpy as np
import pytest

from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


@pytest.mark.parametrize("n,m,g", [(127, 3, 0.5), (129, 70, 0.5), (640, 130, 2.0), (8300, 8, 0.5)])
@pytest.mark.parametrize("stages", [1, 2])
def test_recomputed_pairs_equal_stored(n, m, g, stages):
    p = workloads.mixture(n, m, seed=n + m, gamma=g / m, C=10.0)
    if n < 700:
        i, j = np.triu_indices(n, 1)
    else:   # more tiles than are formed at a time (2145 of 128 x 128)
        rng = np.random.default_rng(n)
        i = rng.integers(0, n - 1, 60000)
        j = rng.integers(i + 1, n)
    order = np.random.default_rng(1).permutation(len(i))
    i, j = i[order], j[order]
    got = {}
    for mode in (gabp.Q_BF16, gabp.Q_RECOMPUTE):
        svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, q_mode=mode, refine=0, stages=stages)
        got[mode] = []
        for k in (0, 1, 3, 20):
            svm.solve(k, 0.0)
            got[mode].append(gabp.svm_get_pairs(svm.h, i, j))
        svm.close()
    for a, b in zip(got[gabp.Q_BF16], got[gabp.Q_RECOMPUTE]):
        np.testing.assert_array_equal(a, b)
    assert np.abs(got[gabp.Q_BF16][-1]).max() > 0
