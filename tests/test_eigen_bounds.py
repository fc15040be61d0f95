"""The eigenvalue bounds of the seed records, run on the host from the kernels' own header.

lo <= lambda_min and hi >= lambda_max are decided exactly, in rationals: S - lo I and
hi I - S are positive semidefinite.  Shapes: random rotations with condition numbers up to
1e12, near-double smallest and largest eigenvalues, multiples of the identity, diagonal
matrices.  Scaling a matrix by a power of two scales its bounds by it, bit for bit, from
2^-90 to 2^90 (determinants from 1e-82 to 1e81; FP32 holds 1e-38 to 3e38)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#define __host__
#define __device__
#define __forceinline__ inline
#include "apd_eig.cuh"
template <int D> static void all(int n, const double *s, double *lo, double *hi) {
    for (int i = 0; i < n; ++i) {
        double m[D][D];
        for (int e = 0; e < D * D; ++e) m[e / D][e % D] = s[i * D * D + e];
        apd::eigen_bounds<D>(m, lo[i], hi[i]);
    }
}
extern "C" void bounds(int dim, int n, const double *s, double *lo, double *hi) {
    if (dim == 3) all<3>(n, s, lo, hi);
    else all<2>(n, s, lo, hi);
}
"""


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    d = tmp_path_factory.mktemp("eig")
    (d / "eig.cpp").write_text(SOURCE)
    lib = str(d / "eig.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2403_03571_gb300", "csrc"), "-o", lib, str(d / "eig.cpp")], check=True)
    fn = ctypes.CDLL(lib).bounds

    def call(S):
        S = np.ascontiguousarray(S, dtype=np.float64)
        lo, hi = np.empty(len(S)), np.empty(len(S))
        p = [a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in (S, lo, hi)]
        fn(S.shape[1], len(S), *p)
        return lo, hi

    return call


def _det(m):
    if len(m) == 1:
        return m[0][0]
    if len(m) == 2:
        return m[0][0] * m[1][1] - m[0][1] * m[1][0]
    return sum((-1) ** j * m[0][j] * _det([r[:j] + r[j + 1:] for r in m[1:]]) for j in range(3))


def _definite(S, shift, sign):
    """sign (S - shift I) is positive semidefinite, exactly (all principal minors >= 0)."""
    D = len(S)
    m = [[sign * (Fraction(float(S[a, b])) - (Fraction(float(shift)) if a == b else 0)) for b in range(D)]
         for a in range(D)]
    sets = [[a for a in range(D) if (k >> a) & 1] for k in range(1, 2 ** D)]
    return all(_det([[m[a][b] for b in s] for a in s]) >= 0 for s in sets)


def _shapes(dim):
    g = np.random.default_rng(dim)
    lam = [np.ones(dim), np.array([1.0, 2.0, 4.0][:dim]), np.array([1.0, 1.0 + 1e-9, 3.0][:dim])]
    for cond in (1.5, 30.0, 1e3, 1e6) + ((1e9, 1e12) if dim == 3 else ()):
        lam += [np.exp(np.log(cond) * g.random(dim)) for _ in range(6)]
        if dim == 3:
            for gap in (0.0, 1e-14, 1e-12, 1e-9, 1e-6, 1e-3):  # near-double smallest, largest
                lam += [np.array([1.0, 1.0 + gap, cond]), np.array([1.0, cond, cond * (1.0 + gap)])]
    S = []
    for v in lam:
        Q = np.linalg.qr(g.standard_normal((dim, dim)))[0]
        m = (Q * (v * np.exp(g.uniform(-0.7, 0.7)))) @ Q.T
        S += [0.5 * (m + m.T), np.diag(v)]
    return np.array(S)


@pytest.mark.parametrize("dim", [2, 3])
def test_bounds_hold_exactly(bounds, dim):
    S = _shapes(dim)
    for k in (-90, -22, 0, 22, 90):
        T = np.ldexp(S, k)
        lo, hi = bounds(T)
        assert np.isfinite(lo).all() and np.isfinite(hi).all()
        for m, a, b in zip(T, lo, hi):
            assert _definite(m, a, 1), (k, m, a)
            assert _definite(m, b, -1), (k, m, b)


@pytest.mark.parametrize("dim", [2, 3])
def test_bounds_are_close_and_scale_exactly(bounds, dim):
    S = _shapes(dim)
    lo, hi = bounds(S)
    ev = np.linalg.eigvalsh(S)
    mild = ev[:, -1] < 2e3 * ev[:, 0]
    # close for the grains in use: within 5 % below, and mean + 2 spread above
    assert np.all(lo[mild] >= 0.95 * ev[mild, 0])
    assert np.all(hi <= 2.0 * ev[:, -1] * (1.0 + 1e-6))
    for k in range(-90, 91, 3):
        a, b = bounds(np.ldexp(S, k))
        assert np.array_equal(a, np.ldexp(lo, k)) and np.array_equal(b, np.ldexp(hi, k)), k
