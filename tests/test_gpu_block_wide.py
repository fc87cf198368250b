"""P^{-1} on an FP32 block so wide that a thread sums U^T V over a thousand rows and more: the sums of 64 rows must not be
lost against a large one before them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_small_sums_behind_a_large_one():
    from paper_2202_11599_gb300 import nysadmm as nx
    d, k = 4096, 4096
    # H = 1 1^T 2^20 + alt alt^T: eigenvectors of entries +-2^-6, exact in FP32
    one, alt = np.ones(d), np.where(np.arange(d) % 2 == 0, 1.0, -1.0)
    A = np.zeros((4, d))
    A[0], A[1] = 1024.0 * one, alt
    Om = np.random.default_rng(0).standard_normal((d, 2))
    P = nx.sketch(nx.Matrix(torch.from_numpy(A).cuda()), torch.from_numpy(Om).cuda())
    U = P.U.float()
    assert torch.equal(U.abs(), torch.full_like(U, 2.0 ** -6))
    # u . v per 64 rows: 2^24, then 1 each; the sums of the alternating eigenvector are those of pairs that cancel but the first
    v = torch.full((d,), 1.0, device="cuda")
    v[:64] = 0.0
    v[0] = 2.0 ** 30
    V = v[:, None].expand(d, k).contiguous()
    rho = 1.0
    Y = P.apply(V, rho)
    lam = P.lam.double()
    c = ((lam[-1] + rho) / (lam + rho) - 1.0).cuda()
    ref = v.double() + U.double() @ (c * (U.double().T @ v.double()))
    # g rounded to FP32 (2^24 and 63 more: +-1) and scaled by U = 2^-6, y rounded once per column of U
    bound = 2.0 ** -6 * 2.0 + 3 * 2.0 ** -24 * ref.abs()
    assert torch.all((Y.double() - ref[:, None]).abs() <= bound[:, None])
