"""Batches without a set plan: no further from 64 bits than with sixteen values a
thread."""
import numpy as np
import pytest

from paper_1007_3470_gb300 import workloads as W
from tests.gpu_helpers import need_gpu
from tests.test_gpu_accuracy import _batch, _error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("projection", [False, True])
@pytest.mark.parametrize("nmin,nmax,count", [(256, 256, 800), (512, 512, 800), (1024, 1024, 300), (2048, 2048, 200),
                                             (128, 4096, 400), (2048, 2048, 20)])
def test_fp32_defaults(projection, nmin, nmax, count):
    """Both runs round as often; 0.5 % for the chance of 3 seeds."""
    need_gpu()
    case = _batch(nmin, count, nmax=nmax, steps=60, projection=projection)
    assert _error(case, range(3)) <= 1.005 * _error(case, range(3), 16)


@pytest.mark.parametrize("nmin,nmax,count", [(128, 128, 60), (512, 512, 60), (1024, 1024, 60), (1024, 1024, 310),
                                             (128, 4096, 40)])
def test_fp64_defaults(nmin, nmax, count):
    """The same transforms in work items of other sizes: the same bits (clusters, which
    arrange them otherwise, have their own test)."""
    need_gpu()
    from paper_1007_3470_gb300 import hfs
    sizes = tuple(n for n in (128, 256, 512, 1024, 2048, 4096) if nmin <= n <= nmax)
    insts, psis, _ = W.batch_1d(count=count, seed=5, sizes=sizes)
    out = []
    for plan in (False, True):
        s = hfs.Solver(insts, precision="c128", chunk_steps=4)
        s.set_schedule(0.01, "strang", hfs.HFS_FLOW_CF4)
        if plan:
            for n in sizes:
                s.set_plan(n, 16)
        s.set_psi(psis)
        s.step(3)
        out.append((s.get_psi(), s.norm(), s.energy()))
        assert s.status() == hfs.HFS_OK
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
