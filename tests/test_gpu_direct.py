"""Tensor-core products that convert A as they read it, at the edges of their tiles (128 and 256 rows,
32-element K steps, the 64 / 128 / 208 / 256 column classes): bit for bit the prepared cp.async form,
in the sketch and in the block matvecs of a regularisation path."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import nys_inputs as gen  # noqa: E402
from paper_2202_11599_gb300 import nysadmm as nx  # noqa: E402


def _forms(monkeypatch, run):
    out = []
    for env in ("1", "0"):
        monkeypatch.setenv("NYS_TC_TMA", env)
        out.append(run())
    return out


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,d,s", [(1, 8, 1), (128, 128, 65), (129, 129, 100), (257, 511, 128), (700, 257, 200),
                                   (4097, 640, 209)])
def test_sketch_bits(monkeypatch, dtype, n, d, s):
    rng = np.random.default_rng(n + s)
    A = rng.standard_normal((n, d)) * gen.column_scales(d, 0.5)[None, :]
    M = nx.Matrix.padded(torch.from_numpy(A).cuda(), dtype)
    Om = torch.from_numpy(gen.gaussian_test_matrix(d, s, n)).cuda()
    D = torch.from_numpy(rng.random(n) + 0.1).cuda()

    def run():
        P = nx.sketch(M, Om, D=D, diag_shift=0.1)
        return P.lam.clone(), P.U.clone()

    a, b = _forms(monkeypatch, run)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,d,k", [(130, 96, 3), (1000, 257, 64), (640, 300, 70)])
def test_path_bits(monkeypatch, dtype, n, d, k):
    p = gen.lasso_problem(n, d, nnz=5, gamma_frac=0.05, seed=d)
    A = nx.Matrix.padded(torch.from_numpy(p.A).cuda(), dtype)
    b = torch.from_numpy(p.b).cuda()
    Om = torch.from_numpy(gen.gaussian_test_matrix(d, 20, d)).cuda()
    gammas = torch.linspace(1.0, 0.1, k, dtype=torch.float64) * p.gamma

    def run():
        out = nx.nysadmm_solve_path(A, b, gammas, 1.0, 20, 1e-6, Om, admm_iters=4, pcg_fixed=[2] * 4)
        return out["X"].clone(), out["Z"].clone()

    a, b2 = _forms(monkeypatch, run)
    assert torch.equal(a[0], b2[0]) and torch.equal(a[1], b2[1])
