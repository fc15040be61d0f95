"""The dual kernel's reduction (64 cells per cluster, 32 columns of clusters, rounds above
the workspace's rows) and the direction's recursion at the edges of both forms (16 pairs
share a warp's halves, 32 seeds a block), against the FP64 oracle.

Tolerances: a cell's terms are a few dozen FP64 operations on the integer moments, whose
second moments cancel against S1 S1 / m; with the trees' depth below 64 operations the
value errs by at most 64 * 1.1e-16 of the terms' magnitudes before cancellation.  The
direction's sums run over n terms in trees of depth log2(n) + n / 4864."""
import numpy as np
import pytest

import oracle
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu
U = 64 * 1.1e-16


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


@pytest.mark.parametrize("dim,n,m", [(2, 1, 12), (3, 3, 8), (2, 4, 16), (3, 5, 12), (2, 63, 32), (3, 64, 16),
                                     (2, 65, 32), (3, 129, 20), (2, 2048, 96), (3, 2049, 32), (2, 4200, 128)])
def test_dual_at_reduction_edges(capi, dim, n, m):
    inst = synth.make_instance(dim, n, m, 5 * n + dim)
    g = np.random.Generator(np.random.PCG64(n))
    w = g.normal(0, 0.1 * n ** (-2.0 / dim), n)
    x, A, wd, v = dev(inst.x), dev(inst.A), dev(w), dev(inst.v)
    ws = capi.Workspace(dim, n, inst.grid.num_pixels)
    mom = torch.zeros((n, 1 + dim + dim * (dim + 1) // 2), dtype=torch.int64, device="cuda")
    capi.apd_cell_moments(inst.grid, x, A, wd, mom, ws)
    out = [torch.zeros(k, dtype=torch.float64, device="cuda") for k in (1, n, 1)]
    capi.apd_dual_value_grad(inst.grid, x, A, wd, v, *out, ws)
    mo = host(mom)
    val, grad, err = oracle.dual_from_moments(inst.grid, inst.x, inst.A, w, inst.v, mo)[:3]
    cell = inst.grid.measure / inst.grid.num_pixels
    span = float(np.max(np.asarray(inst.grid.hi) - np.asarray(inst.grid.lo))) + float(np.abs(inst.x).max())
    terms = np.sum(np.abs(inst.v * w)) + cell * np.sum(mo[:, 0] * (np.abs(w) + span ** 2 * np.abs(inst.A).sum((1, 2))))
    assert abs(float(host(out[0])[0]) - val) <= U * terms
    np.testing.assert_array_equal(host(out[1]), grad)
    assert float(host(out[2])[0]) == pytest.approx(np.max(np.abs(grad) / inst.v), rel=4e-15)


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("n,hist", [(31, 2), (32, 16), (33, 17), (64, 15), (4864, 16), (4865, 18), (9729, 5)])
def test_direction_at_form_edges(capi, n, hist, fused):
    g = np.random.default_rng(3 * n + hist)
    S = g.standard_normal((hist, n))
    Y = S * g.uniform(0.5, 2.0, n) + 0.05 * g.standard_normal((hist, n))
    q = g.standard_normal(n)
    rc, p, gp = capi.apd_lbfgs_check(S, Y, q, fused)
    assert rc == capi.APD_OK
    if fused:
        Y = Y.copy()
        Y[-1] = q - (q - Y[-1])  # the newest pair as the device rounds it
    ref = oracle.lbfgs_direction(S, Y, q, (S[-1] @ Y[-1]) / (Y[-1] @ Y[-1]))
    # two loops of hist steps, each amplifying its dot products' rounding by |s||y| / s.y < 4
    tol = 2 * hist * 4 * U * (np.log2(n) + n / 4864.0)
    assert np.max(np.abs(p - ref)) <= tol * np.max(np.abs(ref))
    assert abs(gp - q @ ref) <= tol * (np.abs(q) @ np.abs(ref))
