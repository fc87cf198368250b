"""The FP64 pass for narrow rows (apass_rows64.cu) against its definition, where its stages, row
groups and column split can go wrong: one row, fewer rows than SMs, one stage and several, a last
group of one to three rows, one column, odd widths, the widest row it takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2202_11599_gb300 import nysadmm as nx  # noqa: E402


@pytest.mark.parametrize("n,d", [(1, 1), (3, 2), (151, 65), (153, 500), (2000, 500), (2001, 501), (5003, 63), (20011, 301),
                                 (3001, 1023), (9001, 2047)])
def test_rows64_pass(n, d):
    rng = np.random.default_rng(n + d)
    A = rng.standard_normal((n, d))
    M = nx.Matrix.padded(torch.from_numpy(A).cuda())
    for w in (None, rng.uniform(0.0, 1.0, n)):
        p = rng.standard_normal(d + 1)
        for off in (0, 1):   # p on and off a 16-byte boundary
            pt = torch.from_numpy(p).cuda()[off:off + d]
            y = nx.hmatvec(M, pt, 0.5, None if w is None else torch.from_numpy(w).cuda()).cpu().numpy()
            ps, ww = p[off:off + d], np.ones(n) if w is None else w
            ref = A.T @ (ww * (A @ ps)) + 0.5 * ps
            mag = np.abs(A).T @ (ww * (np.abs(A) @ np.abs(ps))) + 0.5 * np.abs(ps)
            # a dot product of length d and a sum over n rows, each at most n + d roundings of 2^-53
            assert np.all(np.abs(y - ref) <= 2.0 ** -52 * (np.sqrt(n) + np.sqrt(d) + 8) * mag)


@pytest.mark.parametrize("n,d", [(700, 300), (2001, 501)])
def test_rows64_logistic_and_objective(n, d):
    rng = np.random.default_rng(n)
    A, x = rng.standard_normal((n, d)) / np.sqrt(d), rng.standard_normal(d)
    b = np.sign(rng.standard_normal(n))
    t = A @ x
    f, g, _ = nx.objective("logistic", nx.Matrix.padded(torch.from_numpy(A).cuda()), torch.from_numpy(b).cuda(), 0.1,
                           torch.from_numpy(x).cuda())
    b01 = 0.5 * (1.0 + b)
    ref = np.sum(np.maximum(t, 0) + np.log1p(np.exp(-np.abs(t))) - b01 * t) + 0.1 * np.abs(x).sum()
    grad = A.T @ (1.0 / (1.0 + np.exp(-t)) - b01)
    assert abs(f - ref) <= 1e-12 * abs(ref) and abs(g - np.abs(grad).max()) <= 1e-12 * np.abs(grad).max()
