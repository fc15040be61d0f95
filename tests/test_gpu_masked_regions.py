"""The masked discretisation's region form where its branches change: refinement
factors that divide the tiles or not, up to and past its limit of 16, rows shorter
and longer than a warp's run, windows of one label, boundaries everywhere, and the
64-pixel floor below which the per-pixel form runs.  Coarse labels, refined counts
and fine moments equal the masked oracle's."""
import numpy as np
import pytest

import oracle
from oracle import masked as om
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


@pytest.mark.parametrize("dim,n,res,r", [
    (2, 30, (64, 64), 2), (2, 30, (33, 40), 5), (2, 12, (70, 9), 16), (2, 12, (20, 18), 17), (2, 3, (5, 4), 3),
    (2, 900, (31, 65), 3), (2, 1, (128, 32), 7),
    (3, 20, (16, 16, 16), 2), (3, 40, (33, 12, 17), 3), (3, 6, (9, 8, 10), 7), (3, 3, (8, 8, 8), 16),
    (3, 4, (3, 4, 5), 2), (3, 700, (12, 11, 13), 4), (3, 50, (40, 6, 5), 1),
])
@pytest.mark.parametrize("prune", [False, True])
def test_masked_regions_match_oracle(capi, dim, n, res, r, prune):
    inst = synth.make_instance(dim, n, 8, 300 + n)
    grid = synth.Grid(dim, res)
    g = np.random.Generator(np.random.PCG64(n + r))
    w = 0.3 * g.standard_normal(n) * n ** (-2.0 / dim)
    ws = capi.Workspace(dim, n, grid.num_pixels)
    ws.set_pruning(prune)
    hc, bnd, fine = om.labels(grid, r, inst.x, inst.A, w)
    ref = oracle.moments(om.fine_grid(grid, r), fine, n)
    for _ in range(2):  # the second call starts from the first one's buffers
        mom = torch.full((n, oracle.moment_width(dim)), -1, dtype=torch.int64, device="cuda")
        lab = torch.full((grid.num_pixels,), -1, dtype=torch.int32, device="cuda")
        refined = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        capi.apd_masked_moments(grid, r, dev(inst.x), dev(inst.A), dev(w), mom, lab, ws, refined=refined)
        assert ws.status() == capi.APD_OK
        assert np.array_equal(host(lab), hc)
        assert int(host(refined)[0]) == int(bnd.sum()) * r ** dim
        assert np.array_equal(host(mom), ref), np.argwhere(host(mom) != ref)[:5]
