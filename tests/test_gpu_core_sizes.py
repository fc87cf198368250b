"""The Nystrom core (Cholesky on a cluster, inverse of the factor, eigensolve with its FP32 start and
corrections) at the edges of its forms -- ranks around 8, 64, 128, 224, 320 and 448 -- and on the
spectra an eigensolve meets: graded, exponential, rank-deficient, all eigenvalues equal, clusters."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import nys_inputs as gen  # noqa: E402
import oracle.nysadmm_oracle as o  # noqa: E402
from paper_2202_11599_gb300 import nysadmm as nx  # noqa: E402


def _check(A, s, seed):
    d = A.shape[1]
    Om = gen.gaussian_test_matrix(d, s, seed)
    P = nx.sketch(nx.Matrix.padded(torch.from_numpy(A).cuda()), torch.from_numpy(np.ascontiguousarray(Om)).cuda())
    U, lam, _, _, _ = o.nystrom(lambda X: A.T @ (A @ X), Om, shift_scale=np.sqrt(d))
    got, Ug = P.lam.numpy(), P.U.cpu().numpy()
    assert np.all(np.diff(got) <= 0)
    assert np.max(np.abs(got - lam)) <= 1e-10 * lam[0]
    V = np.random.default_rng(seed).standard_normal((d, 3))
    ref = U @ (lam[:, None] * (U.T @ V))
    assert np.max(np.abs(Ug @ (got[:, None] * (Ug.T @ V)) - ref)) <= 1e-10 * lam[0] * np.max(np.abs(V)) * np.sqrt(d)


@pytest.mark.parametrize("s", [1, 2, 3, 7, 8, 9, 24, 63, 64, 65, 66, 127, 128, 129, 130, 224, 225, 320, 321, 448, 449])
def test_ranks(s):
    d = max(40, s + s // 3)
    rng = np.random.default_rng(s)
    _check(rng.standard_normal((d + 60, d)) * (1.0 + np.arange(d))[None, :] ** -0.8, s, s)


@pytest.mark.parametrize("s", [33, 100, 230])
def test_spectra(s):
    d, n = 2 * s, 3 * s
    Q = gen.orthonormal_columns(n, d, s)
    Z = gen.orthonormal_columns(d, d, s + 1)
    j = np.arange(d)
    for sig in (1.0 / (1.0 + j), 10.0 ** (-j / 8.0), 1.0 / (1.0 + j) ** 2, np.ones(d),
                np.repeat(10.0 ** -np.arange(0.0, 2.5, 0.5), -(-d // 5))[:d], np.where(j < s // 3, 1.0 / (1.0 + j), 0.0)):
        _check((Q * sig) @ Z.T, s, s + 2)
