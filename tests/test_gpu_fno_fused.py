"""The surrogate's fused kernels against the GEMM-by-GEMM path.

The fused forward keeps the operand roundings and the order of accumulation
of the GEMM kernels, so the two paths agree bit for bit.  Below 8192 rows the
tcgen05 setting takes no tensor-core GEMM: it is then the plain GEMM-by-GEMM
path, the reference here.  The sizes are the edges of what the fused kernels
accept: one warp row and eight of them, one mode tile with pad rows (8 modes)
and several, every width, projection widths of one tile and of sixteen, one
output channel and eight, one layer, batches around the 64-sample tile of the
mixing product."""
import numpy as np
import pytest

from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu

# grid, width, modes, layers, in_ch, proj, out_ch
CONFIGS = [(256, 64, 32, 4, 7, 128, 2), (64, 16, 8, 2, 7, 32, 2), (128, 32, 16, 3, 5, 64, 3),
           (256, 64, 64, 1, 8, 16, 1), (32, 16, 16, 2, 1, 256, 8)]


def _model(cfg, batch, seed=0):
    torch = need_gpu()
    from paper_1007_3470_gb300.fno import Fno, FnoConfig
    m = Fno(FnoConfig(*cfg), max_batch=batch, train=True, seed=None)
    rng = np.random.default_rng(seed)
    m.set_params((rng.uniform(-1, 1, m.nparams) / np.sqrt(cfg[1])).astype(np.float32))
    x = rng.standard_normal((batch, cfg[0], cfg[4])).astype(np.float32)
    y = rng.standard_normal((batch, cfg[0], cfg[6])).astype(np.float32)
    return m, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()


@pytest.mark.parametrize("cfg", CONFIGS)
@pytest.mark.parametrize("batch", [1, 31])
def test_forward_equals_gemm_by_gemm(cfg, batch):
    torch = need_gpu()
    from paper_1007_3470_gb300.fno import HFS_FNO_GEMM_TCGEN05
    m, x, _ = _model(cfg, batch)
    fused = m.forward(x)
    m.set_gemm_engine(HFS_FNO_GEMM_TCGEN05)
    plain = m.forward(x)
    assert torch.isfinite(plain).all()
    assert torch.equal(fused, plain)
    m.close()


@pytest.mark.parametrize("batch", [64, 65, 1300])
def test_forward_does_not_depend_on_the_batch(batch):
    """More samples than CTAs and ragged tiles: each sample as in a batch of its own."""
    torch = need_gpu()
    m, x, _ = _model((64, 16, 8, 2, 7, 32, 2), batch)
    whole = m.forward(x)
    assert torch.equal(whole, torch.cat([m.forward(p) for p in x.split(17)]))
    m.close()
