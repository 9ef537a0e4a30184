"""The arithmetic of the plain FP64 CG's A p on isotropic grids, checked on the host: p
truncated to 60-bit fixed point at 2^59 / B, the weighted sum in two 32-bit limbs that
loses its last 8 bits. No limb or sum leaves 64 bits at the largest values, the error
stays within (3264 + 256) units of the copy, and over the directions of a CG it is below
the FP64 stencil's."""
from fractions import Fraction

import numpy as np

IW = [-1470, 270, -27, 2]  # 180 delta^2 lap; 19 weights of 3264 in all


def _fixed(v, e):
    """v 2^(59 - e), truncated towards zero."""
    return np.trunc(np.ldexp(v, 59 - e)).astype(np.int64)


def _weigh(m, s1, s2, s3):
    """-(the weighted sum) / 2^8 as the kernel forms it, in wrapping 64-bit integers."""
    lo = [v & np.int64(0xffffffff) for v in (m, s1, s2, s3)]
    hi = [v >> np.int64(32) for v in (m, s1, s2, s3)]
    h = hi[0] * 1470 - hi[1] * 270 + hi[2] * 27 - hi[3] * 2
    low = lo[0] * 1470 - lo[1] * 270 + lo[2] * 27 - lo[3] * 2
    return (h << np.int64(24)) + (low >> np.int64(8))


def test_extremes_stay_in_64_bits_and_within_the_bound():
    rng = np.random.default_rng(3)
    top = 2 ** 59
    signs = rng.choice([-1, 1], size=(4000, 19))
    vals = signs * np.where(rng.random((4000, 19)) < 0.5, top, rng.integers(0, top, (4000, 19)))
    vals[0], vals[1] = top, -top
    vals[2] = [top] + [-top] * 6 + [top] * 6 + [-top] * 6  # every term of one sign
    vals[3] = -vals[2]
    for v in vals.astype(object):
        s = [int(v[0]), sum(map(int, v[1:7])), sum(map(int, v[7:13])), sum(map(int, v[13:19]))]
        assert max(abs(x) for x in s) < 2 ** 63
        exact = -(IW[0] * s[0] + IW[1] * s[1] + IW[2] * s[2] + IW[3] * s[3])
        out = int(_weigh(*(np.array([x], np.int64) for x in s))[0])
        assert 0 <= exact - 256 * out < 256


def test_error_over_cg_directions():
    """A ball of R_PE 9, a Gaussian charge; exact A p of sampled points in rationals."""
    R, delta = 9, 0.195
    n = 2 * R + 7
    x = np.arange(n) - n // 2
    X, Y, Z = np.meshgrid(x, x, x, indexing="ij")
    ball = X * X + Y * Y + Z * Z <= R * R
    w = [-49 / 18 * 3 / delta ** 2, 1.5 / delta ** 2, -0.15 / delta ** 2, 1 / 90 / delta ** 2]
    s = slice(3, -3)

    def sums(f):
        out = []
        for q in (1, 2, 3):
            t = 0
            for ax in range(3):
                a, b = [s] * 3, [s] * 3
                a[ax], b[ax] = slice(3 + q, n - 3 + q), slice(3 - q, n - 3 - q)
                t = t + (f[tuple(a)] + f[tuple(b)])
            out.append(t)
        return out

    def lap64(f):
        t = sums(f)
        out = np.zeros_like(f)
        out[s, s, s] = w[0] * f[s, s, s] + w[1] * t[0] + w[2] * t[1] + w[3] * t[2]
        return out

    b = np.exp(-3 * delta ** 2 * ((X - 1.3) ** 2 + Y ** 2 + (Z + 0.7) ** 2)) * ball
    r, p = b.copy(), b.copy()
    rr = (r * r).sum()
    d2 = Fraction(delta) ** 2
    pts = np.argwhere(ball)[::37]
    for it in range(41):
        ap = -lap64(p) * ball
        if it % 10 == 0:
            e = int(np.frexp(np.abs(p).max())[1])
            F = _fixed(p, e)
            t = sums(F)
            fx = _weigh(F[s, s, s], *t).astype(np.float64) * 2.0 ** (8 - 59 + e) / (180 * delta ** 2)
            e_fix, e_64 = [], []
            for i, j, k in pts:
                ex = Fraction(0)
                for q in range(4):
                    for o in ([(0, 0, 0)] if q == 0 else [(q, 0, 0), (-q, 0, 0), (0, q, 0), (0, -q, 0), (0, 0, q), (0, 0, -q)]):
                        ex -= IW[q] * Fraction(float(p[i + o[0], j + o[1], k + o[2]]))
                ex /= 180 * d2
                e_fix.append(float(Fraction(float(fx[i - 3, j - 3, k - 3])) - ex))
                e_64.append(float(Fraction(float(ap[i, j, k])) - ex))
            unit = 2.0 ** (e - 59) / (180 * delta ** 2)
            # the truncations, the dropped bits, and the roundings of the conversion and the scale
            assert np.abs(e_fix).max() <= (3264 + 256) * unit + 2.0 ** -51 * np.abs(ap).max()
            assert np.linalg.norm(e_fix) <= np.linalg.norm(e_64), it
        al = rr / (p * ap).sum()
        r = r - al * ap
        rn = (r * r).sum()
        p = (r + rn / rr * p) * ball
        rr = rn
