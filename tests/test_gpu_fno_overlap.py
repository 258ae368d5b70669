"""The surrogate's outputs written over its inputs."""
import ctypes

import pytest

from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers", [1, 2])
@pytest.mark.parametrize("offset", [0, 5000])
def test_forward_over_its_input(layers, offset):
    """The outputs of other samples than a CTA's own lie over inputs that are still to
    be read: the same bits as into a buffer of its own."""
    torch = need_gpu()
    from paper_1007_3470_gb300 import fno as F
    cfg = F.FnoConfig(grid=64, width=32, modes=16, layers=layers, in_ch=7, proj=64, out_ch=2)
    batch = 1000
    m = F.Fno(cfg, max_batch=batch, train=False, seed=3)
    x = torch.randn(batch, 64, 7, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    want = m.forward(x).clone()
    buf = x.clone().reshape(-1)
    out = buf[offset:offset + want.numel()]
    torch.cuda.synchronize()
    assert F._lib().hfs_fno_forward(m.h, ctypes.c_void_p(buf.data_ptr()), ctypes.c_void_p(out.data_ptr()), batch) == 0
    m.stream.synchronize()
    assert torch.equal(out.reshape(want.shape), want)
    m.close()
