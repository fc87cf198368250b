"""A wait of a product that ran out is reported as such, whatever its NaN looks like afterwards."""
import ctypes
import os
import re

import pytest


def test_timeout_comes_first():
    from paper_2202_11599_gb300 import build_lib
    from paper_2202_11599_gb300 import nysadmm as nx
    fn = ctypes.CDLL(build_lib.build()).nys_test_step_status
    for bad in (nx.NYS_EINVAL, nx.NYS_ENOTSPD):
        assert fn(nx.NYS_ETIMEOUT, 0, bad) == nx.NYS_ETIMEOUT
        assert fn(nx.NYS_ETIMEOUT, 1, bad) == nx.NYS_ETIMEOUT
        assert fn(0, 0, bad) == bad
        assert fn(0, 1, bad) == nx.NYS_OK


@pytest.mark.parametrize("name,refusals", [("cholqr2", ["NYS_EINVAL"]), ("nystrom_core", ["NYS_EINVAL", "NYS_ENOTSPD"])])
def test_refusals_of_the_core_ask_the_status_word(name, refusals):
    """The steps that read a product's result back refuse it only through step_status."""
    from paper_2202_11599_gb300 import build_lib
    src = open(os.path.join(build_lib.CSRC, "capi.cu")).read()
    body = re.search(rf"^nys_status {name}\(.*?^}}", src, flags=re.S | re.M).group(0)
    for r in refusals:
        assert re.search(rf"step_status\([^;]*{r}\)", body)
        assert not re.search(rf"return {r};", body)
