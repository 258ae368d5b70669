"""Few instances: warps of a CTA without an instance, and the FP64 phases
(perturbation kinds, off-centre boxes, both splits) against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1007_3470_gb300 import workloads as W
from tests.gpu_helpers import TOL_C64, TOL_C128, budget, need_gpu

pytestmark = pytest.mark.gpu


def _instances(n, count, vi, shift, seed):
    insts, psis, _ = W.batch_1d(count=count, seed=seed, sizes=(n,))
    for inst in insts:
        inst.vi_kind = vi
        if vi == W.VI_X4:
            inst.eps *= 0.01
        if shift:
            inst.a[0] += 0.25
            inst.b[0] += 0.25
    return insts, psis


def _worst(insts, psis, steps, precision, split=0, h=0.005, scheme="strang", **solver):
    from paper_1007_3470_gb300 import hfs
    s = hfs.Solver(insts, precision=precision, chunk_steps=steps, **solver)
    s.set_schedule(h, scheme, hfs.HFS_FLOW_CF4, split=split)
    s.set_psi(psis)
    s.step(steps)
    out = s.split(s.get_psi())
    assert s.status() == hfs.HFS_OK
    s.close()
    for i in insts:
        i.split, i.scheme, i.h, i.ho_flow = split, scheme, h, W.FLOW_CF4
    refs = O.run_batch([O.Problem(**i.as_dict()) for i in insts], psis, steps)
    return max(O.rel_l2(o, r) for o, r in zip(out, refs))


@pytest.mark.parametrize("precision,tol", [("c64", TOL_C64), ("c128", TOL_C128)])
@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("count", [1, 3, 17])
def test_idle_warps(precision, tol, n, count):
    need_gpu()
    insts, psis = _instances(n, count, W.VI_COS, False, seed=n + count)
    assert _worst(insts, psis, 6, precision) <= budget(tol, 0.03)


@pytest.mark.parametrize("vi", [W.VI_NONE, W.VI_X4, W.VI_COS])
@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("split", [0, 1])
def test_fp64_phases(vi, shift, split):
    need_gpu()
    insts, psis = _instances(512, 2, vi, shift, seed=7)
    assert _worst(insts, psis, 6, "c128", split=split, h=0.02, scheme="ni4_82") <= budget(TOL_C128, 0.12)
