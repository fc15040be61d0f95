"""The tiled form of the non-uniform discretisation where its branches change:
labels equal the FP64 oracle's, moments within FP64 summation rounding.

Counts around the rule's floor; one and two dimensions of spread missing; an offset
box; points far outside the seeds and one far outlier; clustered seeds (long lists,
tiles whose list does not fit the store); more seeds than region lists take; exact
ties on a bisector; points that are not finite."""
import numpy as np
import pytest

from oracle import points as op
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


def _run(capi, dim, y, mass, x, A, w):
    n = x.shape[0]
    ws = capi.Workspace(dim, n, 64)
    mom = torch.full((n, op.moment_width(dim)), -5.0, dtype=torch.float64, device="cuda")
    lab = torch.full((y.shape[0],), -1, dtype=torch.int32, device="cuda")
    capi.apd_points_moments(dev(y), dev(mass), dev(x), dev(A), dev(w), mom, ws, labels=lab)
    return ws, host(lab), host(mom)


def _check(capi, dim, y, x, A, w):
    mass = np.random.default_rng(1).uniform(0.5, 1.5, y.shape[0]) / y.shape[0]
    ws, lab, mom = _run(capi, dim, y, mass, x, A, w)
    assert ws.status() == capi.APD_OK
    ref = op.assign(y, x, A, w)
    assert np.array_equal(lab, ref), f"{np.count_nonzero(lab != ref)} labels differ"
    want = op.moments(y, mass, ref, x.shape[0])
    scale = np.abs(want).max(axis=0) + 1e-300
    assert np.all(np.abs(mom - want) <= 1e-12 * scale)


def _seeds(dim, n, seed, lo=0.0, hi=1.0, ws=0.3):
    g = synth.rng(seed)
    x = lo + (hi - lo) * g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n) if dim == 2 else synth.aniso_3d_lognormal(g, n)
    return x, A, ws * g.standard_normal(n) * n ** (-2.0 / dim)


@pytest.mark.parametrize("dim,n,count", [(2, 8, 255), (2, 8, 256), (3, 9, 257), (3, 40, 1000), (2, 700, 40001),
                                         (3, 500, 30011), (3, 33, 3), (2, 3000, 5000), (2, 39, 300), (2, 40, 256),
                                         (3, 11, 300), (3, 12, 256), (2, 8, 48639), (3, 8, 48640), (2, 13, 48641)])
def test_counts(capi, dim, n, count):
    x, A, w = _seeds(dim, n, n)
    _check(capi, dim, np.random.default_rng(count).random((count, dim)), x, A, w)


@pytest.mark.parametrize("dim", [2, 3])
def test_boxes(capi, dim):
    g = np.random.default_rng(3)
    x, A, w = _seeds(dim, 120, 5)
    y = g.random((6000, dim))
    flat = y.copy()
    flat[:, 0] = 0.25  # a line or plane
    _check(capi, dim, flat, x, A, w)
    _check(capi, dim, np.full((700, dim), 0.5), x, A, w)  # one place
    _check(capi, dim, 3.0 * y - 1.0, x, A, w)  # beyond the seeds on all sides
    far = y.copy()
    far[17] = 1e4  # one outlier
    _check(capi, dim, far, x, A, w)
    xo, Ao, wo = _seeds(dim, 120, 6, lo=-300.5, hi=-299.5)
    _check(capi, dim, y - 300.5, xo, Ao, wo)


@pytest.mark.parametrize("dim", [2, 3])
def test_clustered_and_many_seeds(capi, dim):
    g = np.random.default_rng(4)
    x, A, w = _seeds(dim, 1500, 7, lo=0.5, hi=0.51, ws=0.0)
    _check(capi, dim, g.random((4000, dim)), x, A, w)
    x, A, w = _seeds(dim, 16500, 8, ws=0.05)
    _check(capi, dim, g.random((600, dim)), x, A, w)


def test_ties_and_points_that_are_not_finite(capi):
    # equal seeds: every point ties; the lowest index wins
    x, A, w = _seeds(3, 10, 9)
    idx = np.tile(np.arange(10), 4)
    y = np.random.default_rng(5).random((3000, 3))
    _check(capi, 3, y, x[idx], A[idx], w[idx])
    y[100, 1] = np.nan
    y[200, 0] = np.inf
    ws, lab, _ = _run(capi, 3, y, np.full(3000, 1.0), x, A, w)
    assert ws.status() != capi.APD_OK
    ok = np.isfinite(y).all(axis=1)
    assert np.array_equal(lab[ok], op.assign(y[ok], x, A, w))
