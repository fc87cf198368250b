"""U^T w over the blocks of the fused vector steps, FP32 partials: as accurate as FP64 additions in the same order."""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sums(part, c=1.0):
    from paper_2202_11599_gb300 import nysadmm as nx
    fn = nx.lib().nys_test_g_entry
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32, ctypes.c_float, ctypes.c_void_p, ctypes.c_void_p]
    P = torch.from_numpy(np.ascontiguousarray(part, dtype=np.float32)).cuda()
    out = torch.empty(part.shape[1], device="cuda")
    assert fn(P.data_ptr(), part.shape[0], part.shape[1], c, out.data_ptr(), None) == 0
    return out.cpu().numpy()


def test_three_scales_that_cancel():
    # 50 bits from the first to the second value: held by FP64, not by two FP32 words once 2^19 joins them
    v = np.array([2.0 ** 44, 2.0 ** -6, 2.0 ** 19, -2.0 ** 44, -2.0 ** 19])
    assert np.cumsum(v)[-1] == 2.0 ** -6
    assert _sums(np.repeat(v[:, None], 3, axis=1)).tolist() == [2.0 ** -6] * 3


@pytest.mark.parametrize("nb", [1, 16, 31, 33, 79, 304])
def test_random_scales(nb):
    rng = np.random.default_rng(nb)
    part = (rng.standard_normal((nb, 130)) * 2.0 ** rng.integers(-40, 40, (nb, 130))).astype(np.float32)
    got = _sums(part, -0.75).astype(np.float64)
    for i in range(130):
        exact = -0.75 * math.fsum(part[:, i].astype(np.float64))
        mag = float(np.sum(np.abs(part[:, i].astype(np.float64))))
        assert abs(got[i] - exact) <= 2.0 ** -24 * abs(exact) + nb * 2.0 ** -53 * mag


def test_range():
    big = np.array([[3e38, 3e38, np.inf, np.nan], [3e38, -3e38, 1.0, 1.0], [-3e38, 1.0, 1.0, 1.0]])
    out = _sums(big)
    assert out[0] == np.float32(3e38) and out[1] == 1.0 and np.isinf(out[2]) and np.isnan(out[3])
    assert _sums(big, 0.25)[0] == np.float32(np.float32(3e38) * 0.25)
