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


@pytest.mark.parametrize("cfg", CONFIGS)
@pytest.mark.parametrize("batch", [1, 31])
def test_gradients_equal_gemm_by_gemm(cfg, batch):
    """Loss and gradients: the same rounded operands, FP32 sums in another
    order.  A sum of n terms in FP32 differs between two orders by at most
    n 2^-24 of the sum of its terms' magnitudes and by sqrt(n) 2^-24 of their
    root mean square as a rule; with n = 8192 rows at most that is 5.4e-6 of a
    gradient's norm, and a BF16 rounding that falls the other way moves one
    operand in thousands by 2^-8 (about 3e-5 of a norm together)."""
    torch = need_gpu()
    from paper_1007_3470_gb300.fno import HFS_FNO_GEMM_TCGEN05
    m, x, y = _model(cfg, batch)
    loss, g = m.loss_grad(x, y)
    m.set_gemm_engine(HFS_FNO_GEMM_TCGEN05)
    loss_ref, ref = m.loss_grad(x, y)
    assert abs(loss - loss_ref) <= 1e-6 * loss_ref
    assert torch.isfinite(ref).all()
    assert float((g - ref).norm()) <= 5e-5 * float(ref.norm())
    m.close()


def test_gradient_vector_need_not_be_aligned():
    """A gradient vector on a 4-byte boundary that is no 8-byte boundary."""
    torch = need_gpu()
    import ctypes
    from paper_1007_3470_gb300.fno import _lib
    m, x, y = _model(CONFIGS[1], 5)
    _, ref = m.loss_grad(x, y)
    buf = torch.zeros(m.nparams + 1, device="cuda")
    torch.cuda.synchronize()
    vp = ctypes.c_void_p
    assert _lib().hfs_fno_loss_grad(m.h, vp(x.data_ptr()), vp(y.data_ptr()), 5, vp(buf.data_ptr() + 4), None) == 0
    m.stream.synchronize()
    assert float((buf[1:] - ref).norm()) <= 1e-6 * float(ref.norm())
    m.close()


def test_training_steps_follow_the_gemm_by_gemm_path():
    """Adam and the BF16 weight copies: the losses of a short training run on
    either path (steps of 1e-3 on weights near 0.2: a gradient entry whose sign
    is noise moves one weight, the loss by less than 1e-3 of itself)."""
    need_gpu()
    from paper_1007_3470_gb300.fno import HFS_FNO_GEMM_TCGEN05
    losses = []
    for engine in (0, HFS_FNO_GEMM_TCGEN05):
        m, x, y = _model(CONFIGS[2], 9)
        m.set_gemm_engine(engine)
        losses.append([m.train_step(x, y, 1e-3) for _ in range(12)])
        m.close()
    assert losses[0][-1] < losses[0][0]
    assert np.allclose(losses[0], losses[1], rtol=1e-3)
