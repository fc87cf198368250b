"""Accuracy of the FP64 products entry by entry, against exact integer sums: K at the edges of the 32-deep
stages, of the 64-deep steps of the check and of the read-outs, both layouts of A, odd leading dimensions, and
entries whose scales oppose each other, where digits relative to a row's largest entry would lose them.

Bound: that of a chain of FMAs with its partial sums, (K + slices + 2) 2^-53 sum |a||b| with at most K / 64 + 1
slices, for every input.  Rows of one scale and K < 128 (one slice): the digits' own,
2^-53 |c| + 9.2 K 2^-60 2^ea 2^eb, which a wrong digit or order of any weight would exceed."""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import nys_inputs as gen  # noqa: E402
import oracle.nysadmm_oracle as o  # noqa: E402


def _product(A, B, kc, D=None, pad=0):
    """C = diag(D) A B^T on the device; A is M x K and stored as it is (kc) or transposed."""
    from paper_2202_11599_gb300 import nysadmm as nx
    fn = nx.lib().nys_test_gemm64
    i64, ptr = ctypes.c_int64, ctypes.c_void_p
    fn.argtypes = [ptr, ctypes.c_int32, i64, i64, ptr, i64, ctypes.c_int32, i64, ptr, ptr, ptr]
    stored = A if kc else A.T
    dev = []
    for X in (stored, B):
        P = np.full((X.shape[0], X.shape[1] + pad), 7e77)   # the padding is not read as data
        P[:, :X.shape[1]] = X
        dev.append(torch.from_numpy(np.ascontiguousarray(P)).cuda())
    M, N, K = A.shape[0], B.shape[0], A.shape[1]
    C = torch.full((N, M), math.nan, dtype=torch.float64, device="cuda")
    Dd = None if D is None else torch.from_numpy(D).cuda()
    st = fn(dev[0].data_ptr(), int(kc), dev[0].shape[1], M, dev[1].data_ptr(), dev[1].shape[1], N, K,
            None if D is None else Dd.data_ptr(), C.data_ptr(), None)
    assert st == 0
    return C.cpu().numpy().T


def _ints(row, off):
    m, e = np.frexp(row)
    return [int(mm) << int(ee) if ee >= 0 else int(mm) >> int(-ee) for mm, ee in zip(np.ldexp(m, 53).astype(np.int64), e - 53 + off)]


def _check(A, B, C, own_bound=False, samples=250):
    M, N, K = A.shape[0], B.shape[0], A.shape[1]
    off = 53 + int(-min(np.frexp(np.abs(X[X != 0]).min())[1] if np.any(X) else 0 for X in (A, B)))
    off = max(off, 53)
    rng = np.random.default_rng(K)
    S0 = np.abs(A) @ np.abs(B).T
    at = [(int(rng.integers(M)), int(rng.integers(N))) for _ in range(samples)]
    # the outputs whose sum is smallest beside their rows' maxima, and a corner
    rel = S0 / (np.abs(A).max(1)[:, None] * np.abs(B).max(1)[None, :] + 1e-300)
    at += [tuple(int(v) for v in np.unravel_index(i, rel.shape)) for i in np.argsort(rel, axis=None)[:40]] + [(M - 1, N - 1)]
    ia, ib = {}, {}
    for m, n in at:
        a = ia.setdefault(m, _ints(A[m], off))
        b = ib.setdefault(n, _ints(B[n], off))
        exact = sum(x * y for x, y in zip(a, b))
        S = sum(abs(x * y) for x, y in zip(a, b))
        got = C[m, n]
        assert math.isfinite(got)
        num, den = float(got).as_integer_ratio()
        err = abs((num << (2 * off)) // den - exact)
        if own_bound:
            ea, eb = np.frexp(np.abs(A[m]).max())[1] - 1, np.frexp(np.abs(B[n]).max())[1] - 1
            sh = 2 * off - 60 + int(ea) + int(eb)
            lim = (abs(exact) >> 53) + (int(92 * K) << sh) // 10 + 2
        else:
            lim = ((K + K // 64 + 3) * S >> 53) + 2
        assert err <= lim, (m, n, err / max(1, lim))


def _inputs(kind, M, N, K, rng):
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    if kind == "cancel":      # sums that cancel to their last bits
        B[:, 1::2] = -B[:, 0:K - K % 2:2]
        A[:, 1::2] = A[:, 0:K - K % 2:2] * (1 + 1e-13)
    elif kind == "same":      # every digit near its largest, of one sign
        A[:] = B[:] = np.float64(0x3f7f7f7f7f7f7f00) * 2.0 ** -61
    elif kind == "graded":    # rows of very different scale
        A *= 2.0 ** rng.integers(-40, 40, M)[:, None]
        B *= 2.0 ** rng.integers(-40, 40, N)[:, None]
    elif kind == "opposed":   # columns of A against those of B
        t = 2.0 ** rng.integers(-30, 30, K)
        A, B = A * t, B / t
    elif kind == "outlier":   # one column, met by zeros
        A[:, 0] *= 2.0 ** 70
        B[:, 0] = 0.0
    elif kind == "scattered":  # no scaling of K undoes this
        A = A * 2.0 ** rng.integers(-60, 60, (M, K))
        B = B * 2.0 ** rng.integers(-60, 60, (N, K))
    elif kind == "sparse":
        A[rng.random((M, K)) < 0.9] = 0.0
        B[rng.random((N, K)) < 0.5] = 0.0
        A[M // 2] = 0.0
    return A, B


@pytest.mark.parametrize("kc", [True, False])
@pytest.mark.parametrize("M,N,K,pad", [(1, 1, 1, 1), (130, 65, 31, 0), (129, 3, 33, 1), (40, 130, 127, 3)])
@pytest.mark.parametrize("kind", ["normal", "cancel", "same", "graded"])
def test_digits(kind, M, N, K, pad, kc):
    A, B = _inputs(kind, M, N, K, np.random.default_rng(M + K))
    _check(A, B, _product(A, B, kc, pad=pad), own_bound=True)


@pytest.mark.parametrize("kc", [True, False])
@pytest.mark.parametrize("M,N,K,pad", [(1, 1, 2, 0), (130, 65, 65, 1), (33, 20, 513, 2), (260, 9, 1300, 0)])
@pytest.mark.parametrize("kind", ["normal", "opposed", "outlier", "scattered", "sparse", "same"])
def test_any_scale(kind, M, N, K, pad, kc):
    A, B = _inputs(kind, M, N, K, np.random.default_rng(N + K))
    _check(A, B, _product(A, B, kc, pad=pad))


@pytest.mark.parametrize("kc", [True, False])
def test_long_group_of_equal_signs(kc):
    """More tiles than SMs: 256 K in one slice."""
    A, B = _inputs("same", 160 * 128, 64, 256, np.random.default_rng(0))
    _check(A, B, _product(A, B, kc), own_bound=True, samples=2)


@pytest.mark.parametrize("kc", [True, False])
def test_row_factors_and_extremes(kc):
    rng = np.random.default_rng(5)
    A, B = _inputs("normal", 70, 12, 200, rng)
    D = rng.standard_normal(70)
    C, CD = _product(A, B, kc), _product(A, B, kc, D)
    assert np.max(np.abs(CD - D[:, None] * C)) <= 4e-16 * np.max(np.abs(CD))
    _check(A * 2.0 ** -600, B, _product(A * 2.0 ** -600, B, kc), samples=40)
    tiny = A.copy()
    tiny[3] *= 2.0 ** -1060                   # a row of denormals beside ordinary ones
    # 200 products of denormals with ordinary numbers: each rounded to a multiple of 2^-1074
    ref = tiny @ B.T
    assert np.all(np.abs(_product(tiny, B, kc)[3] - ref[3]) <= 200 * 2.0 ** -1074 + 200 * 2.0 ** -53 * np.abs(ref[3]))
    bad = A.copy()
    bad[5, 17], bad[40, 2] = np.inf, np.nan
    got, want = _product(bad, B, kc), bad @ B.T
    assert np.array_equal(np.isfinite(got), np.isfinite(want)) and np.array_equal(np.isnan(got), np.isnan(want))


@pytest.mark.parametrize("bits", [13, 27, 50])
def test_sketch_of_weighted_rows(bits):
    """Rows scaled by s_i with weights 1 / s_i^2 (weighted least squares): H is that of the unscaled rows, exactly for
    powers of two; and a row of any size with weight 0 counts for nothing.  The bound of test_gpu_gemm64.py."""
    from paper_2202_11599_gb300 import nysadmm as nx
    n, d, s = 700, 90, 20
    rng = np.random.default_rng(bits)
    G = rng.standard_normal((n, d))
    G[0] = 0.0
    Om = gen.gaussian_test_matrix(d, s, 3)
    U, lam, _, _, _ = o.nystrom(lambda X: G.T @ (G @ X), Om, shift_scale=np.sqrt(d))
    ref = U @ (lam[:, None] * (U.T @ np.eye(d)))
    sc = 2.0 ** rng.integers(-bits, bits + 1, n)
    for big in (0.0, 2.0 ** (2 * bits)):
        A, D = G * sc[:, None], 1.0 / sc ** 2
        A[0], D[0] = big, 0.0
        P = nx.sketch(nx.Matrix.padded(torch.from_numpy(A).cuda()), torch.from_numpy(np.ascontiguousarray(Om)).cuda(),
                      D=torch.from_numpy(D).cuda())
        got, Ug = P.lam.numpy(), P.U.cpu().numpy()
        assert np.max(np.abs(got - lam)) <= 1e-10 * lam[0]
        assert np.max(np.abs(Ug @ (got[:, None] * Ug.T) - ref)) <= 1e-10 * lam[0] * np.sqrt(d)
