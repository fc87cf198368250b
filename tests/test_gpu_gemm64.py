"""FP64 products on the tensor cores, through the FP64 sketch they carry (Y = A^T D A Omega, the
Gram matrices, U = B V): sizes at the edges of the 128 x 64 tiles, of the 32-deep stages and of the
256-deep read-outs, odd leading dimensions, rows and columns of very different scale, zero rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import nys_inputs as gen  # noqa: E402
import oracle.nysadmm_oracle as o  # noqa: E402


def _check(A, s, seed, D=None):
    from paper_2202_11599_gb300 import nysadmm as nx
    d = A.shape[1]
    Om = gen.gaussian_test_matrix(d, s, seed)
    M = nx.Matrix.padded(torch.from_numpy(A).cuda())
    P = nx.sketch(M, torch.from_numpy(np.ascontiguousarray(Om)).cuda(), D=None if D is None else torch.from_numpy(D).cuda())
    w = np.ones(A.shape[0]) if D is None else D
    U, lam, _, _, _ = o.nystrom(lambda X: A.T @ (w[:, None] * (A @ X)), Om, shift_scale=np.sqrt(d))
    got, Ug = P.lam.numpy(), P.U.cpu().numpy()
    # FP64 rounding of the products and of the core (s up to 130): the bound of the FP64 parity tests
    assert np.max(np.abs(got - lam)) <= 1e-10 * lam[0]
    # U Lam U^T on random vectors (U itself is not unique)
    V = np.random.default_rng(seed).standard_normal((d, 3))
    ref = U @ (lam[:, None] * (U.T @ V))
    assert np.max(np.abs(Ug @ (got[:, None] * (Ug.T @ V)) - ref)) <= 1e-10 * lam[0] * np.max(np.abs(V)) * np.sqrt(d)


@pytest.mark.parametrize("n,d,s", [(40, 31, 1), (127, 33, 2), (129, 65, 63), (300, 128, 64), (513, 257, 65), (1000, 129, 128),
                                   (2050, 511, 130)])
def test_sketch_sizes(n, d, s):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, d)) * (1.0 + np.arange(d))[None, :] ** -0.7
    _check(A, s, d)
    _check(A, s, d + 1, D=rng.uniform(0.01, 0.25, n))


def test_sketch_scales():
    rng = np.random.default_rng(3)
    A = rng.standard_normal((700, 90))
    _check(A * 10.0 ** rng.integers(-12, 4, 700)[:, None], 20, 1)     # rows of very different scale
    _check(A * 10.0 ** rng.integers(-12, 4, 90)[None, :], 20, 2)      # columns of very different scale
    B = A.copy()
    B[::3] = 0.0
    B[:, 7] = 0.0
    _check(B, 20, 3)                                                  # zero rows and a zero column
    _check(A * 1e30, 20, 4)   # the power iteration squares Y^T Y: 1e252, within FP64
    _check(A * 1e-30, 20, 5)
    _check(np.abs(A) + 1.0, 20, 6)                                    # all positive: the sums of equal sign
    _check(np.full((700, 90), 0.99999) + 1e-3 * A, 20, 7)             # top digits all equal
