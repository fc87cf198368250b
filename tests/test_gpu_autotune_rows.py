"""The autotuner of the fused pass times the form that the plan takes by itself, among others it can keep."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,widths", [(torch.float64, [2048, 4266, 4268, 5001, 10000, 12288]), (torch.float32, [1024, 5000, 16000]),
                                          (torch.bfloat16, [2048, 10000]), (torch.float32, [500])])
def test_default_is_among_the_candidates(dtype, widths):
    from paper_2202_11599_gb300 import nysadmm as nx
    fn = nx.lib().nys_test_rows
    for d in widths:
        M = nx.Matrix.padded(torch.zeros(8, d, device="cuda"), dtype)
        rows, planned = (ctypes.c_int32 * 3)(), ctypes.c_int32()
        n = fn(ctypes.byref(M.c), rows, ctypes.byref(planned))
        assert planned.value in list(rows[:n]), (d, list(rows[:n]), planned.value)
        if dtype == torch.float64:
            assert list(rows[:n]) == [1, 2]


def test_tuned_plan_is_a_candidate_that_was_timed():
    from paper_2202_11599_gb300 import nysadmm as nx
    fn = nx.lib().nys_test_rows
    M = nx.Matrix(torch.randn(2000, 6000, dtype=torch.float64, device="cuda"))
    best, ms = nx.autotune_apass(M)
    rows, planned = (ctypes.c_int32 * 3)(), ctypes.c_int32()
    n = fn(ctypes.byref(M.c), rows, ctypes.byref(planned))
    assert n == 2 and planned.value == best and ms > 0


@pytest.mark.parametrize("d", [500, 3000])
def test_rows_too_long_for_a_stage_are_refused(d):
    from paper_2202_11599_gb300 import nysadmm as nx
    A = torch.zeros(3, 13000, dtype=torch.float64, device="cuda")
    m = nx.NysMatrixC(ctypes.c_void_p(A.data_ptr()), nx.NYS_F64, 3, d, 13000)
    assert nx.lib().nys_autotune_apass(ctypes.byref(m), None, None, None) == nx.NYS_EINVAL
