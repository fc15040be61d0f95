"""Points whose box is much larger than the seeds' neighbourhood: two tilings, one of that
neighbourhood and one of the whole box.  Outliers near and far, seeds in one place, two
groups of points, points that do not meet the seeds, points on the neighbourhood's edge:
labels equal the FP64 oracle's, moments within FP64 summation rounding."""
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


def _check(capi, dim, y, x, A, w):
    n = x.shape[0]
    mass = np.random.default_rng(1).uniform(0.5, 1.5, y.shape[0]) / y.shape[0]
    ws = capi.Workspace(dim, n, 64)
    mom = torch.full((n, op.moment_width(dim)), -5.0, dtype=torch.float64, device="cuda")
    lab = torch.full((y.shape[0],), -1, dtype=torch.int32, device="cuda")
    for _ in range(2):  # the second call starts from the first one's tilings
        capi.apd_points_moments(dev(y), dev(mass), dev(x), dev(A), dev(w), mom, ws, labels=lab)
        assert ws.status() == capi.APD_OK
    ref = op.assign(y, x, A, w)
    assert np.array_equal(host(lab), ref), f"{np.count_nonzero(host(lab) != ref)} labels differ"
    want = op.moments(y, mass, ref, n)
    assert np.all(np.abs(host(mom) - want) <= 1e-12 * (np.abs(want).max(axis=0) + 1e-300))


@pytest.mark.parametrize("dim,n,count", [(2, 60, 3000), (3, 60, 3001), (2, 900, 20000), (3, 900, 20000), (3, 12, 256),
                                         (2, 300, 50000)])
def test_wide_boxes(capi, dim, n, count):
    g = synth.rng(n + count)
    x = g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n) if dim == 2 else synth.aniso_3d_lognormal(g, n)
    w = 0.3 * g.standard_normal(n) * n ** (-2.0 / dim)
    y = g.random((count, dim))
    for far in (4.5, 50.0, -1e3, 1e6):  # one outlier
        z = y.copy()
        z[count // 2] = far
        _check(capi, dim, z, x, A, w)
    z = y.copy()
    z[7, 0], z[8, dim - 1] = 30.0, -200.0  # on single axes
    _check(capi, dim, z, x, A, w)
    _check(capi, dim, y, 0.1 * x, A, 0.01 * w)  # seeds in a corner
    _check(capi, dim, y, 0.5 + 1e-3 * x, A, 1e-6 * w)  # seeds in one place inside
    z = y.copy()
    z[::2] += 300.0  # two groups
    _check(capi, dim, z, x, A, w)
    _check(capi, dim, 100.0 * y + 40.0, x, A, w)  # none near the seeds
    z = -5.0 + 11.0 * y
    edge = [x.min(axis=0) - 0.5 * np.ptp(x, axis=0).max(), x.max(axis=0) + 0.5 * np.ptp(x, axis=0).max()]
    z[:50] = edge[0]
    z[50:100] = edge[1]
    z[100:120] = np.nextafter(edge[1], 10.0)
    _check(capi, dim, z, x, A, w)
