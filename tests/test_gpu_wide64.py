"""FP64 pass for wide rows: row blocks that do and do not fill a CTA's warps, one row, odd widths (the
last vector half outside the matrix), every count of column vectors per thread from two to twelve,
every row mode's result against torch in FP64 (plain, weighted, transposed only)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2202_11599_gb300 import nysadmm as nx  # noqa: E402

EPS = 2.0 ** -53


@pytest.mark.parametrize("n,d", [(1, 2048), (3, 2049), (151, 3072), (153, 3073), (2432, 4097), (2433, 5121),
                                 (4865, 6145), (700, 7169), (700, 8193), (700, 9217), (700, 10241), (300, 11265),
                                 (300, 12287), (5000, 2050)])
@pytest.mark.parametrize("rows", [None, "1"])
def test_against_torch(monkeypatch, n, d, rows):
    if rows:
        monkeypatch.setenv("NYS_APASS_ROWS", rows)
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 31 + d)
    ld = d + 1 + (d & 1) * 2 + 1 & ~1
    T = torch.full((n, ld), float("nan"), dtype=torch.float64, device="cuda")   # what lies beyond a row stays out
    T[:, :d] = torch.randn(n, d, generator=g, device="cuda", dtype=torch.float64)
    A = T[:, :d]
    p = torch.randn(d, generator=g, device="cuda", dtype=torch.float64)
    D = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) + 0.1
    M = nx.Matrix(A)
    a = A.abs()
    for w in (None, D):
        t = A @ p
        ref = A.T @ (t if w is None else w * t) + 0.5 * p
        # n + d products and sums, each rounded once, in either computation
        mag = a.T @ ((a @ p.abs()) * (1.0 if w is None else w)) + 0.5 * p.abs()
        y = nx.hmatvec(M, p, 0.5, w)
        assert bool(((y - ref).abs() <= 2 * (n + d + 8) * EPS * mag).all())
        assert torch.equal(y, nx.hmatvec(M, p, 0.5, w))
