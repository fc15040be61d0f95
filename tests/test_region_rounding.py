"""The pruned scorer's rounding where it is largest: tiles far from their region's centre,
seeds near those tiles.  Restated in numpy FP32; a position difference is compared with the
exact rational one, a pixel's value with the FP64 costs (whose own error is 2^-29 of the
bound's unit).  With u = 2^-24, off the tile's offset and r its half-width:

    |d - exact| <= 3 u |d| + 4 u |off| + 4 u 2^-24 (|x| + |y|_max),
    |value - exact| <= k u (S_i + S_a + |dw| + 2^-24 (|w_i| + |w_a|)), k = 33 (3D), 43 (2D),

which the scorer's 64 u covers with a third to spare in 2D, half in 3D.  The pixels' FP32
steps are those of test_region_bounds."""
from fractions import Fraction

import numpy as np
import pytest

from test_region_bounds import U, _local, _pair

f32 = np.float32
TILE = {2: (32, 16), 3: (8, 8, 8)}
REGION = {2: (64, 64), 3: (16, 16, 16)}
UNITS = {2: 43.0, 3: 33.0}


def _tiles(dim):
    return [tuple(int(t) for t in np.unravel_index(k, [r // t for r, t in zip(REGION[dim], TILE[dim])]))
            for k in range(int(np.prod([r // t for r, t in zip(REGION[dim], TILE[dim])])))]


def _setup(dim, seed, tc, shift, spread):
    g = np.random.default_rng(seed)
    res = int(g.integers(70, 900))
    h = 1.0 / res
    T, R = np.array(TILE[dim]), np.array(REGION[dim])
    rb = np.array([int(g.integers(0, res // r)) * r for r in R])
    c64 = shift + (rb + R / 2) * h
    off64 = (np.array(tc) * T + T / 2 - R / 2) * h
    x = c64 + off64 + spread * h * g.standard_normal((80, dim))  # around the tile's centre
    h32 = f32(h)
    off = ((np.array(tc) * T + T / 2 - R / 2).astype(f32) * h32).astype(f32)
    rr = (f32(0.5) * (T - 1).astype(f32) * h32 * f32(1 + 2.0 ** -22)).astype(f32)
    return g, h, h32, rb, c64, off, rr, x, f32(abs(shift) + 1.0)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("shift", [0.0, -7.5, 100.0])
def test_position_differences(dim, shift):
    u = Fraction(1, 2 ** 24)
    worst = 0.0
    for seed in range(4):
        for tc in _tiles(dim):
            g, h, h32, rb, c64, off, rr, x, ymax = _setup(dim, seed, tc, shift, 12.0)
            ch, cl = _pair(c64)
            xh, xl = _pair(x)
            d = (((ch - xh) + (cl - xl)) + off).astype(f32)
            for i in range(0, 80, 7):
                for a in range(dim):
                    n = tc[a] * TILE[dim][a] + TILE[dim][a] // 2 - REGION[dim][a] // 2
                    exact = Fraction(float(c64[a])) + n * Fraction(h) - Fraction(float(x[i, a]))
                    err = abs(Fraction(float(d[i, a])) - exact)
                    bound = u * (3 * abs(exact) + 4 * abs(n * Fraction(h)) +
                                 4 * u * (abs(Fraction(float(x[i, a]))) + Fraction(float(ymax))))
                    assert err <= bound, (seed, tc, i, a)
                    p = u * (abs(exact) + Fraction(float(rr[a])))
                    worst = max(worst, float(err / p))
    assert worst > (5.0 if dim == 2 else 1.0)  # five roundings of p do not cover 2D


@pytest.mark.parametrize("dim", [2, 3])
def test_values(dim):
    worst = 0.0
    T = np.array(TILE[dim])
    for seed in range(6):
        for tc in _tiles(dim):
            for spread in (0.3, 3.0, 20.0):
                g, h, h32, rb, c64, off, rr, x, ymax = _setup(dim, 50 + seed, tc, 0.0, spread)
                n = len(x)
                Q = np.linalg.qr(g.standard_normal((n, dim, dim)))[0]
                A = np.einsum("nij,nj,nkj->nik", Q, np.exp(g.standard_normal((n, dim))), Q)
                A = 0.5 * (A + A.transpose(0, 2, 1))
                w = (spread * h) ** 2 * g.standard_normal(n)
                ch, cl = _pair(c64)
                xh, xl = _pair(x)
                wh, wl = _pair(w)
                A32 = A.astype(f32)
                q, S, hh = _local(dim, ch, cl, off, rr, xh, xl, A32, ymax)
                axes = [(rb[a] + tc[a] * T[a] + np.arange(T[a]) + 0.5) * h for a in range(dim)]
                y = np.stack([m.ravel() for m in np.meshgrid(*axes, indexing="ij")], 1)
                e = np.stack([m.ravel() for m in np.meshgrid(*[((np.arange(t) - t // 2).astype(f32) + f32(0.5)) * h32
                                                               for t in T], indexing="ij")], 1).astype(f32)
                dd = y[:, None, :] - x[None]
                exact = np.einsum("pna,nab,pnb->pn", dd, A, dd) - w
                a = int(np.argmin(q - wh))
                dw = ((wh - wh[a]) + (wl - wl[a])).astype(f32)
                d0 = ((q - q[a]) - dw).astype(f32)
                G = (f32(2) * (hh - hh[a])).astype(f32)
                dA = (A32 - A32[a]).astype(f32)
                unit = (S.astype(np.float64) + S[a] + np.abs(dw) + U * (np.abs(wh) + np.abs(wh[a]))) * float(U)
                f1 = e[:, 1]
                for i in range(0, n, 3):
                    if i == a:
                        continue
                    if dim == 3:
                        f2 = e[:, 2]
                        b = (f32(2) * dA[i, 0, 2] * f2 + (f32(2) * dA[i, 0, 1] * f1 + G[i, 0])).astype(f32)
                        t1 = (f32(2) * dA[i, 1, 2] * f2 + (dA[i, 1, 1] * f1 + G[i, 1])).astype(f32)
                        t2 = (dA[i, 2, 2] * f2 + G[i, 2]).astype(f32)
                        aa = (f2 * t2 + (f1 * t1 + d0[i]).astype(f32)).astype(f32)
                    else:
                        b = (f32(2) * dA[i, 0, 1] * f1 + G[i, 0]).astype(f32)
                        aa = (f1 * (dA[i, 1, 1] * f1 + G[i, 1]).astype(f32) + d0[i]).astype(f32)
                    v = ((dA[i, 0, 0] * e[:, 0] + b).astype(f32) * e[:, 0] + aa).astype(f32)
                    err = np.abs(v.astype(np.float64) - (exact[:, i] - exact[:, a]))
                    worst = max(worst, float(err.max() / unit[i]))
    assert worst <= UNITS[dim], worst
    assert worst > 0.5  # the cases reach the bound's order
