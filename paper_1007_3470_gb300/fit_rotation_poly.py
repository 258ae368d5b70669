"""Fit the polynomials of the FP32 small rotation (kSin*, kCos* in
csrc/hfs_phase.cuh): sin(theta) = theta + theta^3 P(theta^2) with P of degree 2
and cos(theta) - 1 = theta^2 Q(theta^2) with Q of degree 3 on |theta| <= pi/4.

Method: Lawson's algorithm (iteratively reweighted least squares, which
converges to the minimax solution) on Chebyshev nodes, minimising the
relative error; the coefficients are then rounded to FP32 one at a time, the
later ones refitted to the residual after each rounding.

fit64() gives those of the FP64 rotation by f turns, |f| <= 1/8 (kSinF*, kCosF*):
sin(2 pi f) = f (2 pi + f^2 Q(f^2)) with 2 pi as kTwoPi64 + kTwoPi64Lo and
cos(2 pi f) = 1 + f^2 P(f^2), by Remez's exchange in 40 digits (mpmath), the
coefficients rounded to FP64 in the same way.

Run as a script to print the coefficients and the errors of the rounded sets."""
import numpy as np


def _nodes(m=4000, margin=2e-7):
    a = (np.pi / 4) * (1 + margin)
    th = a * np.cos((np.arange(m) + 0.5) * np.pi / m)
    return th[th > 0]


def _lawson(basis, target, den, iters=400):
    w = np.ones_like(target)
    c = None
    for _ in range(iters):
        sw = np.sqrt(w) / den
        c, *_ = np.linalg.lstsq(basis * sw[:, None], target * sw, rcond=None)
        err = np.abs((basis @ c - target) / den)
        w = w * err
        w /= w.sum()
    return c


def fit():
    th = _nodes()
    s = th * th
    sin_t = (np.sin(th) - th) / th ** 3          # P(s)
    cm1 = -2.0 * np.sin(th / 2) ** 2             # cos(theta) - 1 without cancellation
    cos_t = cm1 / s                              # Q(s)
    out = []
    for target, den, npow in ((sin_t, np.sin(th) / th ** 3, 3), (cos_t, np.abs(cos_t), 4)):
        fixed = []
        for k in range(npow):
            resid = target - sum(c * s ** j for j, c in enumerate(fixed))
            basis = np.stack([s ** j for j in range(k, npow)], axis=1)
            fixed.append(float(np.float32(_lawson(basis, resid, den)[0])))
        out.append(fixed)
    return out


def errors(sin_c, cos_c, n=200001):
    th = np.linspace(1e-4, np.pi / 4 * (1 + 2e-7), n)
    s = th * th
    p = th + th ** 3 * np.polyval(list(reversed(sin_c)), s)
    q = s * np.polyval(list(reversed(cos_c)), s)
    cm1 = -2.0 * np.sin(th / 2) ** 2
    return float(np.max(np.abs(p / np.sin(th) - 1))), float(np.max(np.abs(q / cm1 - 1)))


def _targets64():
    """(function of x = f^2, weight of its error, number of coefficients): the
    error of the sine relative, that of the cosine absolute."""
    from mpmath import cos, mp, mpf, pi, sin
    hi = 2 * pi
    two_pi = (float(hi), float(hi - mpf(float(hi))))

    def sin_q(x):
        f = mp.sqrt(x)
        return (sin(2 * pi * f) / f - mpf(two_pi[0]) - mpf(two_pi[1])) / x

    def sin_w(x):
        f = mp.sqrt(x)
        return x * f / sin(2 * pi * f)

    return two_pi, ((sin_q, sin_w, 6), (lambda x: (cos(2 * pi * mp.sqrt(x)) - 1) / x, lambda x: x, 7))


def _range64():
    from mpmath import mpf
    return mpf(10) ** -10, (mpf(1) / 8 * (1 + mpf(2) ** -20)) ** 2


def _remez(fun, weight, n):
    from mpmath import cos, lu_solve, matrix, pi
    lo, hi = _range64()
    grid = [lo + (hi - lo) * (1 - cos(pi * k / 300)) / 2 for k in range(301)]
    pts = [(lo + hi) / 2 - (hi - lo) / 2 * cos(pi * (2 * k + 1) / (2 * (n + 1))) for k in range(n + 1)]
    for _ in range(8):
        A, b = matrix(n + 1, n + 1), matrix(n + 1, 1)
        for i, x in enumerate(pts):
            for j in range(n):
                A[i, j] = x ** j
            A[i, n] = (-1) ** i / weight(x)
            b[i] = fun(x)
        c = list(lu_solve(A, b))[:n]
        err = [weight(x) * (sum(c[j] * x ** j for j in range(n)) - fun(x)) for x in grid]
        # the largest error of every run of one sign
        runs = [[(abs(err[0]), grid[0])]]
        for k in range(1, len(grid)):
            if (err[k] > 0) != (err[k - 1] > 0):
                runs.append([])
            runs[-1].append((abs(err[k]), grid[k]))
        if len(runs) < n + 1:
            break
        pts = sorted(p[1] for p in sorted(map(max, runs), reverse=True)[:n + 1])
    return c


def fit64():
    """((kTwoPi64, kTwoPi64Lo), [kSinF3, ...], [kCosF2, ...])"""
    from mpmath import mp, mpf
    with mp.workdps(40):
        two_pi, targets = _targets64()
        out = []
        for fun, weight, n in targets:
            fixed = []
            for k in range(n):
                def rest(x):
                    return (fun(x) - sum(mpf(v) * x ** j for j, v in enumerate(fixed))) / x ** k
                fixed.append(float(_remez(rest, lambda x: weight(x) * x ** k, n - k)[0]))
            out.append(fixed)
        return two_pi, out[0], out[1]


def errors64(coefficients, n=2000):
    """Largest errors of the rounded sets, exactly evaluated: (sin, relative; cos)."""
    from mpmath import mp, mpf
    with mp.workdps(40):
        lo, hi = _range64()
        xs = [lo + (hi - lo) * k / n for k in range(n + 1)]
        return tuple(float(max(abs(w(x) * (sum(mpf(v) * x ** j for j, v in enumerate(c)) - fun(x))) for x in xs))
                     for (fun, w, _), c in zip(_targets64()[1], coefficients))


if __name__ == "__main__":
    sc, cc = fit()
    print("sin:", ["%.9e" % c for c in sc])
    print("cos-1:", ["%.9e" % c for c in cc])
    print("relative errors (sin, cos-1): %.3e %.3e" % errors(sc, cc))
    two_pi, s64, c64 = fit64()
    print("2 pi:", two_pi)
    print("sin:", s64)
    print("cos:", c64)
    print("errors (sin relative, cos): %.2e %.2e" % errors64((s64, c64)))
