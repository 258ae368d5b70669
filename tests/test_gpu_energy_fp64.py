"""The energy of complex128 states whose perturbation dominates it."""
import numpy as np
import pytest

from paper_1007_3470_gb300 import workloads as W
from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,plan", [(128, 16), (128, 8), (256, 16), (256, 8), (1024, 16), (2048, 8), (4096, 16)])
@pytest.mark.parametrize("step", [0.001, 1.0, 3.139])
def test_perturbation_energy(n, plan, step):
    """One point each of instances with eps = 1e6, everywhere in the box, k T dx =
    `step` (T threads hold points T apart; a recurrence over them is worst near 0 and
    pi), other kinds, whose k is
    not read, between them.  eps cos(k x) is off by the rounding of k x as a sum
    of two products, 2 2^-53 (|k x_t| + |k T e dx|) |sin k x|, and by 2^-53 times: 2 for
    each sine or cosine, 1 for each product, the sum of products and the sum of terms,
    8 in all.  The other terms are exact to 1e-14 of their size (12 passes of the
    transform, 2 2^-53 each, twice for the square)."""
    need_gpu()
    from paper_1007_3470_gb300 import hfs
    T, u, eps, half = n // plan, 2.0 ** -53, 1e6, 16.0
    dx = 2 * half / n
    k = step / (T * dx)
    insts, psis, want, bound = [], [], [], []
    points = [e * T + t for e in range(plan) for t in (0, T // 2, T - 1)]
    for i, j in enumerate(points + [0, n // 3, n - 1]):
        kind = W.VI_COS if i < len(points) else (W.VI_NONE, W.VI_X4, W.VI_NONE)[i - len(points)]
        insts.append(W.Instance(n=[n], a=[-half], b=[half], w0=1.0, eps=eps if kind == W.VI_COS else 1e-3, vi_kind=kind,
                                vi_k=k if kind == W.VI_COS else np.nan, sigma=2.0))
        psi = np.zeros(n, dtype=np.complex128)
        psi[j] = (0.6 - 0.8j) / np.sqrt(dx)
        psis.append(psi)
        L = np.longdouble
        d = L(psi[j].real) ** 2 + L(psi[j].imag) ** 2
        x = L(-half) + L(dx) * j
        vi = {W.VI_COS: L(eps) * np.cos(L(k) * x), W.VI_X4: L(1e-3) * x ** 4, W.VI_NONE: L(0)}[kind]
        m = np.fft.fftfreq(n, 1.0 / n).astype(L)
        kin = d * ((2 * L(np.pi) + L(1.2246467991473532e-16) * 2) / L(2 * half)) ** 2 * np.sum(m * m) / (2 * n)
        rest = kin + (L(0.5) * x * x + d) * d
        want.append(dx * (rest + vi * d))
        t = j % T
        arg = abs(k * (t - n // 2) * dx) + abs(k * (j - t) * dx)
        cos_err = eps * u * (2 * arg * abs(np.sin(float(k * x))) + 8) if kind == W.VI_COS else 1e-14 * abs(vi)
        bound.append(dx * (d * cos_err + 1e-14 * rest))
    order = np.random.default_rng(1).permutation(len(insts))
    s = hfs.Solver([insts[i] for i in order], precision="c128", chunk_steps=4)
    s.set_plan(n, plan)
    s.set_psi([psis[i] for i in order])
    got = s.energy()
    s.close()
    for i, e in zip(order, got):
        assert abs(np.longdouble(e) - want[i]) <= bound[i], (i, float(abs(e - want[i]) / bound[i]))
