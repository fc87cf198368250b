"""The Cholesky factor and the product with its inverse, entry by entry against longer arithmetic (numpy's long
double): pivots over the whole exponent range, both forms of the factorisation, panels whose columns differ in scale."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53
LD = np.longdouble


def _run(M, Y=None):
    from paper_2202_11599_gb300 import nysadmm as nx
    fn = nx.lib().nys_test_triangular
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_int64, ctypes.POINTER(ctypes.c_int32), ctypes.c_void_p]
    Md = torch.from_numpy(np.ascontiguousarray(M.T)).cuda()
    Yd = None if Y is None else torch.from_numpy(np.ascontiguousarray(Y.T)).cuda()
    info = ctypes.c_int32(-1)
    st = fn(Md.data_ptr(), M.shape[0], None if Y is None else Yd.data_ptr(), 0 if Y is None else Y.shape[0], ctypes.byref(info), None)
    assert st == 0
    return info.value, Md.cpu().numpy().T, None if Y is None else Yd.cpu().numpy().T


def test_pivots_of_every_exponent():
    """C_kk of a diagonal matrix: the library's reciprocal root is within an ulp (2 u), the product adds u."""
    vals = [np.ldexp(m, e) for e in range(-1070, 1020, 19) for m in (1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52)]
    vals = np.array(vals + [5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0), 2.0 ** -1000, np.nextafter(2.0 ** -1000, 0), 1.7e308])
    for e in (-1000, -2, -1, 0, 1, 2, 3, 4):   # beside powers of two and four
        vals = np.append(vals, [np.nextafter(2.0 ** e, 0), 2.0 ** e, np.nextafter(2.0 ** e, 9e9)])
    for part in np.array_split(vals, 2):
        info, C, _ = _run(np.diag(part))
        assert info == 0
        assert np.array_equal(C, np.diag(np.diag(C)))
        assert np.max(np.abs(np.diag(C) / np.sqrt(part.astype(LD)) - 1)) <= 3 * U


@pytest.mark.parametrize("s", [1, 9, 64, 200, 448, 449])
def test_factor(s):
    rng = np.random.default_rng(s)
    A = rng.standard_normal((s + 20, s)) * 10.0 ** rng.uniform(-4, 4, s)
    M = A.T @ A
    M = 0.5 * (M + M.T)
    info, C, _ = _run(M)
    assert info == 0 and np.array_equal(C, np.triu(C))
    # |C^T C - M| <= gamma_{s+1} |C|^T |C|, with the reciprocal root's ulp and a product in the place of a division
    R = C.T.astype(LD) @ C.astype(LD) - M.astype(LD)
    assert np.max(np.abs(R) / (np.abs(C).T @ np.abs(C))) <= (s + 4) * U


@pytest.mark.parametrize("d,s", [(33, 1), (33, 7), (300, 64), (513, 65), (140, 130)])
@pytest.mark.parametrize("kind", ["plain", "scaled", "dependent"])
def test_times_inverse(kind, d, s):
    """Columns of B = Y C^-1 against the same in long double: the inverse's residual |C x - e| <= (s + 2) u |C||x|, the
    product's 9.1 s 2^-60 times the largest entries of the rows of Y and of the columns of X once Y's columns are
    brought to C's scale, and a rounding."""
    rng = np.random.default_rng(d * s)
    Y = rng.standard_normal((d, s))
    if kind == "scaled":
        Y = Y * 2.0 ** rng.integers(-30, 31, s)
    elif kind == "dependent" and s > 1:
        Y[:, -1] = Y[:, 0] + 1e-5 * Y[:, -1]
    base = Y if d >= s else rng.standard_normal((s, s))
    info, C, B = _run(base.T @ base, Y)
    assert info == 0
    Cl = C.astype(LD)
    X = np.zeros((s, s), dtype=LD)
    for j in range(s):          # back substitution, column j
        x = np.zeros(s, dtype=LD)
        x[j] = 1
        for i in range(j, -1, -1):
            x[i] = (x[i] - Cl[i, i + 1:j + 1] @ x[i + 1:j + 1]) / Cl[i, i]
        X[:, j] = x
    exact = Y.astype(LD) @ X
    aY, aX, aC = np.abs(Y), np.abs(X).astype(np.float64), np.abs(C)
    t = 2.0 ** (np.frexp(aC.max(0))[1] - 1)
    lim = (1.1 * (s + 2) * U * np.linalg.norm(aY @ (aX @ (aC @ aX)), axis=0)
           + 9.2 * s * 2.0 ** -60 * np.linalg.norm((aY / t).max(1)) * (aX * t[:, None]).max(0)
           + U * np.linalg.norm(B, axis=0))
    err = np.linalg.norm((B - exact).astype(np.float64), axis=0)
    assert np.all(err <= lim), np.max(err / lim)
