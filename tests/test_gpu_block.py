"""P^{-1} on a block of vectors (nys_precond_apply) against its definition in FP64, at the edges of
its column forms (1, 2, <= 4, <= 16, more) and of its tiles of rows, ranks and columns."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import nys_inputs as gen  # noqa: E402


def _precond(n, d, s, seed):
    from paper_2202_11599_gb300 import nysadmm as nx
    p = gen.lasso_problem(n, d, seed=seed)
    return nx.sketch(nx.Matrix.padded(torch.from_numpy(p.A).cuda()), torch.from_numpy(gen.gaussian_test_matrix(d, s, seed)).cuda())


@pytest.mark.parametrize("d,s", [(257, 1), (300, 63), (1025, 64), (2051, 130)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_apply_block(d, s, dtype):
    from paper_2202_11599_gb300 import nysadmm as nx
    P = _precond(2 * d, d, s, d)
    U, lam, rho = P.U.cpu().numpy(), P.lam.numpy(), 0.7
    rng = np.random.default_rng(s)
    eps = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -53
    for k in (1, 2, 3, 4, 5, 16, 17, 64, 65, 130):
        V = torch.from_numpy(rng.standard_normal((d, k))).to(dtype)
        Vd = V.double().numpy()
        ref = Vd + U @ (((lam[-1] + rho) / (lam + rho) - 1.0)[:, None] * (U.T @ Vd))
        Y = P.apply(V.cuda(), rho).double().cpu().numpy()
        # rounding of U and c, a dot product of length d and a chain of s + 1 terms, all against
        # the sums of absolute values
        mag = np.abs(Vd) + np.abs(U) @ (np.abs(U).T @ np.abs(Vd))
        assert np.max(np.abs(Y - ref) / mag) <= eps * (6 + 2 * np.sqrt(d) + s), (k, np.max(np.abs(Y - ref) / mag))
        # in place: Y may be V
        W = V.T.contiguous().cuda()
        st = nx.lib().nys_precond_apply(P.h, rho, ctypes.c_void_p(W.data_ptr()), ctypes.c_void_p(W.data_ptr()), k,
                                        nx.NYS_F64 if dtype == torch.float64 else nx.NYS_F32,
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == nx.NYS_OK
        assert np.array_equal(W.T.double().cpu().numpy(), Y)
