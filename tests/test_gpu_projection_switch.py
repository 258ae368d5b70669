"""Work lists that the norm projection's switch leaves alone."""
import numpy as np
import pytest

from paper_1007_3470_gb300 import workloads as W
from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu


def _capture(s, what):
    import torch
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(s.stream):
        graph.capture_begin(capture_error_mode="thread_local")
        what()
        graph.capture_end()
    return graph


@pytest.mark.parametrize("switched_inside", [False, True])
def test_projection_switch_and_captured_steps(switched_inside):
    """A caller's captured step keeps its plans when the projection is switched
    after it; the switch itself is a host call and may be part of a capture.  512
    points take other plans under the projection."""
    torch = need_gpu()
    from paper_1007_3470_gb300 import hfs
    insts, psis, _ = W.batch_1d(count=700, seed=6, sizes=(128, 512, 1024))

    def solver():
        s = hfs.Solver(insts, precision="c64", chunk_steps=4)
        s.set_schedule(0.01, "strang", hfs.HFS_FLOW_CF4)
        s.set_psi(psis)
        return s

    s = solver()
    if switched_inside:
        graph = _capture(s, lambda: (s.set_norm_projection(True), s.step(3)))
    else:
        graph = _capture(s, lambda: s.step(3))
        s.set_norm_projection(True)
    with torch.cuda.stream(s.stream):
        graph.replay()
    got = s.get_psi()
    assert s.status() == hfs.HFS_OK
    # the switch holds for later calls
    s.set_time(0.0)
    s.set_psi(psis)
    s.step(3)
    projected = s.get_psi()
    s.close()
    for project, out in ((switched_inside, got), (True, projected)):
        r = solver()
        r.set_norm_projection(project)
        r.step(3)
        assert np.array_equal(out, r.get_psi())
        r.close()
