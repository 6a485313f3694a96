"""The step headers' logarithms and quotients against plain IEEE operations:
every argument of the logarithms (2^24 and 2^32), every 11-bit pair of the short
quotient, and for every binary32 divisor random dividends and those whose
quotients lie closest to a rounding boundary."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    from paper_2605_00479_gb300 import build
    so = str(tmp_path_factory.mktemp("arithmetic") / "arithmetic_check.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-cudart", "shared",
                           "-I", build.CSRC, os.path.join(HERE, "arithmetic_check.cu"), "-o", so])
    torch.cuda.init()
    fn = ctypes.CDLL(so).check_arithmetic
    fn.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def run(which):
        n = torch.zeros(2, dtype=torch.int64, device="cuda")
        assert fn(which, n.data_ptr(), n.data_ptr() + 8) == 0
        return [int(v) for v in n.cpu()]

    return run


@pytest.mark.parametrize("which", ["logs_24", "logs_32", "logs_64", "quotients_short"])
def test_equal_to_plain_operations(check, which):
    assert check(["logs_24", "logs_32", "logs_64", "quotients_short"].index(which))[0] == 0


def test_quotients(check):
    bad, hard = check(4)
    assert bad == 0
    assert hard > 2**24      # close cases found: several a divisor
