"""A workspace's scratch for point sets is the tensor-core passes' own: its creation takes
no more device memory for them, and calls of both kinds alternate on one workspace."""
import numpy as np
import pytest

import oracle
from oracle import points as op
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


def test_memory_of_a_small_workspace():
    require_gpu()
    from paper_2403_03571_gb300 import capi
    capi.Workspace(3, 10, 64).close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ws = capi.Workspace(3, 1000, 256)
    used = free - torch.cuda.mem_get_info()[0]
    ws.close()
    # 1025 tiles of 16 KB operands, 0.6 MB of lists and headers, under 2 MB of seed data,
    # in about thirty allocations that share 2 MB pages
    assert used <= 24 << 20, used


@pytest.mark.parametrize("dim,n,res", [(2, 500, (200, 150)), (3, 500, (48, 40, 36))])
def test_points_and_tensor_core_passes_alternate(dim, n, res):
    require_gpu()
    from paper_2403_03571_gb300 import capi
    g = synth.rng(5 + dim)
    x = g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n, 0.1) if dim == 2 else synth.aniso_3d_lognormal(g, n, 0.1)
    w = 0.3 * g.standard_normal(n) * n ** (-2.0 / dim)
    grid = synth.Grid(dim, res)
    y = g.random((6000, dim))
    want, pts = oracle.assign(grid, x, A, w), op.assign(y, x, A, w)
    xd, Ad, wd, yd = dev(x), dev(A), dev(w), dev(y)
    mass = torch.full((6000,), 1.0 / 6000, dtype=torch.float64, device="cuda")
    ws = capi.Workspace(dim, n, grid.num_pixels)
    v = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    sols = []
    for prune, prec, inc in ((False, capi.APD_TC_TF32, 1), (True, capi.APD_TC_BF16, 2), (True, capi.APD_TC_TF32, 2)):
        ws.set_pruning(prune)
        ws.set_incremental(inc)
        for _ in range(2):
            lab = torch.full((grid.num_pixels,), -1, dtype=torch.int32, device="cuda")
            capi.apd_assign(grid, xd, Ad, wd, lab, ws, precision=prec)
            assert np.array_equal(host(lab), want)
            pl = torch.full((6000,), -1, dtype=torch.int32, device="cuda")
            mom = torch.empty((n, op.moment_width(dim)), dtype=torch.float64, device="cuda")
            capi.apd_points_moments(yd, mass, xd, Ad, wd, mom, ws, labels=pl)
            assert np.array_equal(host(pl), pts)
            out = torch.zeros(n, dtype=torch.float64, device="cuda")
            capi.apd_solve_weights(grid, xd, Ad, torch.zeros_like(out), v, out, ws,
                                   capi.solve_opts(eps=1e-9, max_evals=6, precision=prec))
            sols.append(host(out))
    assert ws.status() == capi.APD_OK
    for s in sols[1:]:  # the same labels, moments and steps whichever scorer ran
        assert np.array_equal(s, sols[0])
