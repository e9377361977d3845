"""Memory and rounds that outlive one call: handles made and closed by several
threads and streams share the kept blocks, and a chunk of rounds gives the
same bits whether it is launched directly or from its graph."""
import threading

import numpy as np
import pytest

from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


def _train(p, **opts):
    svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, **opts)
    alpha, _, _ = svm.solve(60, 1e-6)
    out = np.array(alpha), np.array(svm.decision(p.X[:30]))
    svm.close()
    return out


@pytest.mark.parametrize("ns", [(130, 257, 640), (40, 300, 1025)])
def test_handles_of_several_threads_share_the_kept_memory(ns):
    ps = [workloads.mixture(n, 5, seed=n) for n in ns]
    want = [_train(p) for p in ps]
    got, errors = {}, []

    def work(k):
        try:
            for r in range(4):
                got[k, r] = _train(ps[(k + r) % len(ps)])
        except Exception as e:   # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (k, r), (alpha, dec) in got.items():
        a, d = want[(k + r) % len(ps)]
        assert np.array_equal(alpha, a) and np.array_equal(dec, d)
    gabp.batch_release()
    assert np.array_equal(_train(ps[1])[0], want[1][0])


@pytest.mark.parametrize("opts", [{}, {"stages": 3}, {"q_mode": gabp.Q_BF16, "refine": 4}])
def test_rounds_launched_directly_and_from_a_graph_agree(opts):
    """The first chunks of a handle are launched one kernel at a time, later
    ones from a captured graph, kept over refits."""
    p, o = (workloads.mixture(700, 6, seed=s) for s in (1, 2))
    ref = {id(x): _train(x, **opts)[0] for x in (p, o)}
    svm = gabp.GabpSVM(p.X, p.y, p.gamma, p.C, **opts)
    for k in range(8):
        x = (p, o)[k % 2]
        svm.refit(x.X, x.y, x.gamma, x.C)
        assert np.array_equal(np.array(svm.solve(60, 1e-6)[0]), ref[id(x)]), k
    svm.close()
