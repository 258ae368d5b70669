"""The complex64 32^3 and 64^3 kernels (a plane pass and a z-pass per sub-stage)
against the FP64 line passes on the device, which the oracle tests pin: every
perturbation kind, calls of one sub-stage and of several schedule chunks (the
first and last plane passes of a call differ), with and without graphs."""
import numpy as np
import pytest

from paper_1007_3470_gb300 import workloads as W
from tests.gpu_helpers import TOL_C64, budget, need_gpu

pytestmark = pytest.mark.gpu


def _run(inst, psi0, precision, graphs, scheme):
    from paper_1007_3470_gb300 import hfs
    s = hfs.Solver([inst], dim=3, precision=precision, chunk_steps=2)
    s.set_schedule(inst.h, scheme, hfs.HFS_FLOW_CF4)
    s.set_graphs(graphs)
    s.set_psi(psi0.ravel())
    for k in (1, 5, 2):
        s.step(k)
    out = s.get_psi()
    assert s.status() == hfs.HFS_OK
    s.close()
    return out.astype(np.complex128)


@pytest.mark.parametrize("n", [32, 64])
@pytest.mark.parametrize("vi", [W.VI_NONE, W.VI_X4, W.VI_COS])
@pytest.mark.parametrize("graphs,scheme", [(False, "strang"), (True, "ni4_82")])
def test_cube_matches_fp64(n, vi, graphs, scheme):
    need_gpu()
    inst, psi0, _ = W.gpe_3d(n=n, h=0.005)
    inst.vi_kind = vi
    if vi == W.VI_X4:
        inst.eps = 1e-3
    inst.b[1], inst.a[1] = 10.0, -10.0  # another mesh width along y
    out = _run(inst, psi0, "c64", graphs, scheme)
    ref = _run(inst, psi0, "c128", graphs, scheme)
    assert np.linalg.norm(out - ref) <= budget(TOL_C64, 0.04) * np.linalg.norm(ref)
