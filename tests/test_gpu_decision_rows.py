"""Decisions of many rows (several slabs of 2^17, workspaces that are kept, grow or
are too large to keep) against FP64, and of rows that are refused: the caller's
output is then as it was.

Bar: as in test_gpu_decision.py, 1e-5 of sum_j |alpha_j y_j| (an FP32 kernel entry
is off by a few units of 2^-24 (1 + gamma (|x|^2 + |z|^2)), gamma |x|^2 < 12 here).
"""
import numpy as np
import pytest

from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu

BAR = 1e-5
SLAB = 1 << 17


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


def _reference(X, y, alpha, gamma, lam, Z):
    X, w = X.astype(np.float64), alpha.astype(np.float64) * y
    out = np.empty(len(Z))
    for a in range(0, len(Z), 8192):
        z = Z[a:a + 8192].astype(np.float64)
        d2 = np.maximum((z * z).sum(1)[:, None] + (X * X).sum(1)[None] - 2.0 * z @ X.T, 0.0)
        out[a:a + 8192] = (np.exp(-gamma * d2) + lam * lam) @ w
    return out, np.abs(w).sum()


def _fit(p, dev):
    torch = pytest.importorskip("torch")
    svm = (gabp.GabpSVM(torch.from_numpy(p.X).cuda(), torch.from_numpy(p.y).cuda(), p.gamma, p.C) if dev
           else gabp.GabpSVM(p.X, p.y, p.gamma, p.C))
    alpha = svm.solve(30, 0.0)[0]
    return svm, (alpha.cpu().numpy() if dev else np.array(alpha)), svm.stats()["lambda_"]


def _rows(Z, t):
    return np.ascontiguousarray(Z[np.arange(t) % len(Z)])


@pytest.mark.parametrize("dev", [False, True])
@pytest.mark.parametrize("m,ts", [(3, (SLAB, SLAB + 129)), (130, (100, 20001, 70001, 100, 2 * SLAB + 1))])
def test_many_rows(m, ts, dev):
    torch = pytest.importorskip("torch")
    p = workloads.mixture(300, m, seed=m)
    svm, alpha, lam = _fit(p, dev)
    base = workloads.test_points(p, 997, seed=5)
    want, scale = _reference(p.X, p.y, alpha, p.gamma, lam, base)
    for t in ts:
        Z = _rows(base, t)
        got = svm.decision(torch.from_numpy(Z).cuda() if dev else Z)
        got = got.cpu().numpy() if dev else np.asarray(got)
        assert got.shape == (t,)
        assert np.max(np.abs(got - want[np.arange(t) % len(base)])) <= BAR * scale, t
    svm.close()


@pytest.mark.parametrize("dev", [False, True])
@pytest.mark.parametrize("t,bad", [(1, 0), (300, 7), (300, 299), (SLAB + 200, 5), (SLAB + 200, SLAB + 150)])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_refused_row_leaves_the_output(t, bad, value, dev):
    torch = pytest.importorskip("torch")
    p = workloads.mixture(300, 4, seed=2)
    svm, _, _ = _fit(p, dev)
    good = _rows(workloads.test_points(p, 500, seed=6), t)
    Z = good.copy()
    Z[bad, 2] = value
    if dev:
        Z, out = torch.from_numpy(Z).cuda(), torch.full((t,), 123.0, device="cuda")
    else:
        out = np.full(t, 123.0, dtype=np.float32)
    want = svm.decision(torch.from_numpy(good).cuda() if dev else good)   # (leaves its values in the workspace)
    with pytest.raises(gabp.GabpError, match=f"test row {bad}:") as e:
        gabp.svm_decision(svm.h, Z, out)
    assert e.value.status == gabp.EINVAL
    assert bool((out == 123.0).all())
    again = svm.decision(torch.from_numpy(good).cuda() if dev else good)
    assert bool((again == want).all())
    svm.close()


# the largest of the small tiles (one 128 x 128 tile fewer than SMs either way, and
# one more) and of the scratch
@pytest.mark.parametrize("n,t", [(151 * 128, 128), (128, 151 * 128), (152 * 128, 127), (127, 152 * 128 + 1), (1, 349525), (1_039_000, 1)])
def test_noalloc_at_its_limits(n, t):
    torch = pytest.importorskip("torch")
    p = workloads.mixture(1000, 3, seed=n % 97)
    X, y = p.X[np.arange(n) % p.n], p.y[np.arange(n) % p.n]
    base = workloads.test_points(p, 61, seed=t % 89)
    alpha = np.random.default_rng(7).random(n, dtype=np.float32) / n
    out = torch.full((t,), float("nan"), device="cuda")
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X, y, alpha, _rows(base, t))]
    gabp.decision_noalloc(*args, p.gamma, 0.25, out)
    w = np.zeros(p.n)
    np.add.at(w, np.arange(n) % p.n, alpha.astype(np.float64) * y)
    want, _ = _reference(p.X, np.ones(p.n), w, p.gamma, 0.25, base)
    scale = np.abs(alpha.astype(np.float64) * y).sum()
    assert np.max(np.abs(out.cpu().numpy() - want[np.arange(t) % len(base)])) <= BAR * scale


def test_wide_rows_need_no_more_memory_than_they_take():
    """2^17 rows of 8000 features (4.2 GB) with 5.5 GB left on the device: the three
    planes of all of them at once would take 6.3."""
    torch = pytest.importorskip("torch")
    n, m, t = 300, 8000, SLAB
    p = workloads.mixture(n, m, seed=9, gamma=0.2 / m)
    svm, alpha, lam = _fit(p, True)
    X = torch.from_numpy(p.X).cuda()
    g = torch.Generator(device="cuda").manual_seed(3)
    Z = X[torch.arange(t, device="cuda") % n]
    Z[:, ::7] += 0.5 * torch.randn((t, len(range(0, m, 7))), device="cuda", generator=g)
    torch.cuda.empty_cache()
    gabp.batch_release()
    filler = torch.empty(max(0, torch.cuda.mem_get_info()[0] - int(5.5e9)), dtype=torch.uint8, device="cuda")
    try:
        got = svm.decision(Z).cpu().numpy()
    finally:
        del filler
        torch.cuda.empty_cache()
    rows = np.unique(np.concatenate([np.arange(0, t, 4001), [t - 1]]))
    want, scale = _reference(p.X, p.y, alpha, p.gamma, lam, Z[torch.from_numpy(rows).cuda()].cpu().numpy())
    assert np.max(np.abs(got[rows] - want)) <= BAR * scale
    svm.close()
