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


def test_fp64_rotation_keeps_the_modulus_for_all_turns(check):
    """|u| = 1 (to a rounding of its squares, 2e-16) from 2^-1000 to 2^1023.9 turns: c^2
    + s^2 and the products round five times at 1 (1.1e-16 each)."""
    assert check("turns_modulus") <= 2e-16 + 2 * 5 * 1.1e-16


@pytest.mark.parametrize("plan", [0, 16, 8])
@pytest.mark.parametrize("sigma", [1e18, 1e25, 1e40])
def test_fp64_state_of_an_absurd_interaction_keeps_its_norm(plan, sigma):
    """Phases beyond 2^49 turns have no angle left, but the step stays unitary
    (two steps: 1e-14)."""
    need_gpu()
    import numpy as np

    from paper_1007_3470_gb300 import hfs
    from paper_1007_3470_gb300 import workloads as W
    insts, psis, _ = W.batch_1d(count=2, seed=3, sizes=(256,))
    for inst in insts:
        inst.sigma = sigma
    s = hfs.Solver(insts, precision="c128", chunk_steps=4)
    s.set_schedule(0.01, "strang", hfs.HFS_FLOW_CF4)
    if plan:
        s.set_plan(256, plan)
    s.set_psi(psis)
    before = s.norm()
    s.step(2)
    assert s.status() == hfs.HFS_OK
    assert np.all(np.abs(s.norm() / before - 1) <= 1e-14)
    s.close()


def test_gelu_over_all_inputs(check):
    """Equal to the accurate function rounded to BF16 but for -0, where it gives +0."""
    assert check("gelu_differences") == 1
