"""Decision values at the edges of the tiles, against FP64: the handle's
(tensor-core Gram, split sums) for every input type and kind of pointer, and the
allocation-free call's two tile sizes.

Bar: an FP32 kernel entry exp(-gamma d2) is off by at most a few units of
2^-24 (1 + gamma (|x|^2 + |z|^2)), below 1e-5 for this data (gamma |x|^2 < 12), and
a decision by that much of sum_j |alpha_j y_j|.
"""
import numpy as np
import pytest

from paper_0810_1648_gb300 import gabp, workloads

pytestmark = pytest.mark.gpu

BAR = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_0810_1648_gb300 import build as gbuild
    gbuild.build()


def _reference(X, y, alpha, gamma, lam, Z):
    X, Z, w = X.astype(np.float64), Z.astype(np.float64), alpha.astype(np.float64) * y
    d2 = np.maximum((Z * Z).sum(1)[:, None] + (X * X).sum(1)[None] - 2.0 * Z @ X.T, 0.0)
    return (np.exp(-gamma * d2) + lam * lam) @ w, np.abs(w).sum()


@pytest.mark.parametrize("n,m", [(127, 5), (129, 64), (700, 65), (1400, 130)])
@pytest.mark.parametrize("dtype", ["f32", "f64", "bf16"])
def test_handle_decision(n, m, dtype):
    torch = pytest.importorskip("torch")
    p = workloads.mixture(n, m, seed=n + m)
    X = torch.from_numpy(p.X).cuda()
    if dtype == "bf16":
        X = X.bfloat16()
    Xh = X.float().cpu().numpy()
    host = Xh.astype(np.float64) if dtype == "f64" else Xh
    dev = dtype == "bf16"
    svm = gabp.GabpSVM(X if dev else host, torch.from_numpy(p.y).cuda() if dev else p.y, p.gamma, p.C)
    alpha = svm.solve(30, 0.0)[0]
    alpha = alpha.cpu().numpy() if dev else np.asarray(alpha)
    lam = svm.stats()["lambda_"]
    for t in (1, 127, 128, 129, 513):
        Z = torch.from_numpy(workloads.test_points(p, t, seed=t))
        Z = Z.bfloat16() if dev else Z
        Zh = Z.float().numpy()
        got = svm.decision(Z.cuda() if dev else Zh.astype(host.dtype))
        got = got.cpu().numpy() if dev else np.asarray(got)
        want, scale = _reference(Xh, p.y, alpha, p.gamma, lam, Zh)
        assert np.max(np.abs(got - want)) <= BAR * scale, t
    svm.close()


@pytest.mark.parametrize("n,t", [(1, 1), (63, 65), (64, 64), (129, 127), (2049, 64), (5000, 400), (3000, 1025)])
@pytest.mark.parametrize("m", [3, 16, 33])
def test_noalloc_decision(n, t, m):
    torch = pytest.importorskip("torch")
    p = workloads.mixture(max(n, 40), m, seed=n)
    X, y, Z = p.X[:n], p.y[:n], workloads.test_points(p, t, seed=t)
    alpha = np.random.default_rng(n).random(n, dtype=np.float32) / n
    out = torch.full((t,), float("nan"), device="cuda")
    gabp.decision_noalloc(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X, y, alpha, Z)), p.gamma, 0.25, out)
    want, scale = _reference(X, y, alpha, p.gamma, 0.25, Z)
    assert np.max(np.abs(out.cpu().numpy() - want)) <= BAR * scale


@pytest.mark.parametrize("m", [8, 64, 12])
@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_rows_off_the_load_alignment(m, dtype):
    """Device rows that begin one element past a 16-byte boundary (the wide
    loads do not apply) give the bits of aligned ones: handle, decision and the
    batched form, which reads FP32 rows in place."""
    torch = pytest.importorskip("torch")
    p = workloads.mixture(300, m, seed=m)
    dt = getattr(torch, dtype)
    Xa = torch.from_numpy(p.X).cuda().to(dt)
    Za = torch.from_numpy(workloads.test_points(p, 140, seed=3)).cuda().to(dt)
    y = torch.from_numpy(p.y).cuda()

    def shifted(t):
        buf = torch.zeros(t.numel() + 1, dtype=dt, device="cuda")
        v = buf[1:].view(t.shape)
        v.copy_(t)
        assert v.data_ptr() % 16
        return v

    outs = []
    for X, Z in ((Xa, Za), (shifted(Xa), shifted(Za))):
        svm = gabp.GabpSVM(X, y, p.gamma, p.C)
        alpha = svm.solve(20, 0.0)[0].clone()
        dec = svm.decision(Z).clone()
        svm.close()
        both = gabp.batch_solve([workloads.Problem(X, y, p.gamma, c) for c in (p.C, 2.0)], 20, 0.0)[0]
        outs.append((alpha, dec, both[0].clone(), both[1].clone()))
    for a, b in zip(*outs):
        assert torch.equal(a, b)
