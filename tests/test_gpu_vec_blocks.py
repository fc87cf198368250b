"""PCG / ADMM vector steps at the edges of their block sizes (one block, one cluster of up to eight,
a cooperative grid, chunks of 64, 128 and 256 elements): the device loop with its fused kernels
against the host-driven loop of separate kernels, bit for bit, and both against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import nys_inputs as gen  # noqa: E402
import oracle.nysadmm_oracle as o  # noqa: E402
from paper_2202_11599_gb300 import nysadmm as nx  # noqa: E402


@pytest.mark.parametrize("n,d,s", [(90, 40, 8), (300, 64, 9), (400, 65, 20), (700, 513, 33), (2300, 2048, 24),
                                   (2300, 2049, 24)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_device_loop_is_the_host_loop(n, d, s, dtype):
    _loops(n, d, s, dtype)


def test_device_loop_is_the_host_loop_wide():
    _loops(300, 19457, 5, torch.float32)   # wider than an FP64 matrix may be


def _loops(n, d, s, dtype):
    p = gen.lasso_problem(n, d, nnz=5, gamma_frac=0.05, seed=d)
    Om = torch.from_numpy(np.ascontiguousarray(gen.gaussian_test_matrix(d, s, d))).cuda()
    A = nx.Matrix.padded(torch.from_numpy(p.A).cuda(), dtype)
    b = torch.from_numpy(p.b).cuda()
    K = 12
    fixed = [k % 4 for k in range(K)]   # iterations with and without PCG steps
    for kw in ({"pcg_fixed": fixed}, {}):
        args = ("lasso", A, b, p.gamma, 1.0, s, 1e-6 if dtype == torch.float64 else 1e-3, Om)
        host = nx.nysadmm_solve(*args, admm_iters=K, device_loop=False, z_trace=True, **kw)
        dev = nx.nysadmm_solve(*args, admm_iters=K, hx_refresh=0, z_trace=True, **kw)
        for f in ("x", "z", "z_trace"):
            assert torch.equal(host[f], dev[f]), (f, kw)
        assert host["info"]["pcg_iters_total"] == dev["info"]["pcg_iters_total"]
        assert host["info"]["r_p"] == dev["info"]["r_p"] and host["info"]["r_d"] == dev["info"]["r_d"]
    if dtype == torch.float64 and d <= 2049:
        ref = o.lasso_nysadmm(p.A, p.b, p.gamma, 1.0, gen.gaussian_test_matrix(d, s, d), K, pcg_tol=1e-10)
        dev = nx.nysadmm_solve("lasso", A, b, p.gamma, 1.0, s, 1e-10, Om, admm_iters=K, pcg_fixed=ref["trace"]["pcg_iters"])
        assert np.linalg.norm(dev["z"].cpu().numpy() - ref["z"]) <= 1e-9 * max(1.0, np.linalg.norm(ref["z"]))
