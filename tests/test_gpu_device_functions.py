"""Device functions over their whole ranges (device_functions.cu)."""
import os
import subprocess

import pytest

from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    need_gpu()
    from paper_1007_3470_gb300 import build as B
    exe = str(tmp_path_factory.mktemp("device") / "device_functions")
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", f"-I{B.INCLUDE}", f"-I{B.CSRC}",
                    os.path.join(HERE, "device_functions.cu"), "-o", exe], check=True, capture_output=True)
    return lambda what: float(subprocess.run([exe, what], check=True, capture_output=True, text=True).stdout)


def test_fp64_rotation_against_sincospi(check):
    """apply_turns: two roundings at the size of the sine or cosine and the
    polynomials' 4e-18, below 2e-16; sincospi's own error is at most 2 ulp of a
    result up to 1 (2.2e-16)."""
    assert check("turns_error") <= 2e-16 + 2.2e-16
