"""FP64 sketches of steep spectra, where only sweeps from the identity keep the small eigenpairs: rows scaled by powers of two
up to 2^+-20 (eigenvalues from 1e-12 to 1e13), and columns decaying like j^-2 at rank 200."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 2])
def test_pcg_on_scaled_rows(seed):
    """H has rank 100 and the preconditioner all of it: what PCG is left with are the pairs' errors (about 20 iterations
    with relatively accurate small pairs, no convergence in 300 with pairs accurate to eps lam_1)."""
    from paper_2202_11599_gb300 import nysadmm as nx
    n, d, s = 100, 210, 100
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    A = torch.randn(n, d, dtype=torch.float64, device="cuda", generator=g)
    A = A * 2.0 ** torch.randint(-20, 21, (n, 1), generator=g, device="cuda").double()
    Om = torch.randn(d, s, dtype=torch.float64, device="cuda", generator=g)
    M = nx.Matrix.padded(A)
    P = nx.sketch(M, Om)
    b = torch.randn(d, dtype=torch.float64, device="cuda", generator=g)
    _, it, _ = nx.pcg_solve(M, b, 2.0, P, tol=1e-8, maxit=100)
    assert it < 100


def test_orthonormal_factor():
    """Columns i and j of U are orthogonal to (what is left of the rotated B^T B at i, j) / (sigma_i sigma_j), at most
    s u lam_1 / lam_s when that is rounding."""
    from paper_2202_11599_gb300 import nysadmm as nx
    n, d, s = 4000, 1000, 200
    g = torch.Generator("cuda")
    g.manual_seed(5)
    A = torch.randn(n, d, dtype=torch.float64, device="cuda", generator=g) * (1.0 + torch.arange(d, device="cuda").double()) ** -2
    Om = torch.randn(d, s, dtype=torch.float64, device="cuda", generator=g)
    P = nx.sketch(nx.Matrix(A), Om)
    U, lam = P.U, P.lam
    ratio = float(lam[-1] / lam[0])
    assert 1e-11 < ratio < 1e-8
    assert (U.T @ U - torch.eye(s, device="cuda")).abs().max().item() <= s * 2.0 ** -53 / ratio
