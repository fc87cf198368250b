"""FP64 pass over wide rows with one to a few rows per CTA, where several warps share a row: against the FP64 definition,
at the row counts around which the sharing changes (for 152 SMs), odd widths, with and without weights."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [2048, 4001, 12288])
@pytest.mark.parametrize("n", [1, 100, 153, 304, 400, 608, 700, 1216, 1300])
def test_few_rows(n, d):
    from paper_2202_11599_gb300 import nysadmm as nx
    g = torch.Generator("cuda")
    g.manual_seed(n * d)
    A = torch.randn(n, d, dtype=torch.float64, device="cuda", generator=g)
    p = torch.randn(d, dtype=torch.float64, device="cuda", generator=g)
    M = nx.Matrix.padded(A)
    for D in (None, torch.rand(n, dtype=torch.float64, device="cuda", generator=g)):
        y = nx.hmatvec(M, p, 0.3, D)
        assert torch.equal(y, nx.hmatvec(M, p, 0.3, D))
        w = 1.0 if D is None else D
        ref = A.T @ (w * (A @ p)) + 0.3 * p
        scale = A.abs().T @ (w * (A.abs() @ p.abs())) + 0.3 * p.abs()
        # the bound of test_gpu_apass.py
        assert ((y - ref).abs() / scale).max().item() <= 1e-12
