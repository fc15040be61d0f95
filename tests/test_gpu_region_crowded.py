"""The pruned scorer where cells are smaller than a few pixels or seeds crowd: lists beyond
a warp's 48 polynomials, beyond the tile's and the region's own lists (their lengths follow
the number of regions), and grids left to the FP32 kernel (more than 4096 seeds on fewer
than 2.5 pixels a seed).  Labels, moments and the slabs' sums equal the FP64 oracle's; a
solve takes the steps of the solver without pruning."""
import numpy as np
import pytest

import oracle
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, instance_tensors, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


def _inst(dim, n, res, hi=1.0, wscale=0.3, copies=1):
    g = synth.rng(n + 3)
    x = hi * g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n, 0.3) if dim == 2 else synth.aniso_3d_lognormal(g, n, 0.3)
    w = wscale * hi ** 2 * g.standard_normal(n) * n ** (-2.0 / dim)
    idx = np.tile(np.arange(n), copies)
    return synth.Instance(synth.Grid(dim, res), x[idx], A[idx], w[idx], np.full(len(idx), 1.0 / len(idx)))


CASES = [
    (3, 900, (20, 18, 16), 1.0, 1), (2, 1500, (70, 66), 1.0, 1),    # tiles past the buffer
    (3, 3000, (24, 20, 18), 1.0, 1), (2, 4000, (90, 80), 1.0, 1),   # regions past their list
    (3, 4200, (17, 16, 33), 1.0, 1), (2, 5000, (64, 65), 1.0, 1),   # left to the FP32 kernel
    (3, 9000, (40, 36, 35), 0.3, 1), (2, 9000, (300, 200), 0.2, 1),  # crowded in a corner
    (2, 4000, (700, 300), 0.1, 1), (3, 4000, (96, 96, 64), 0.2, 1),  # long tile lists on 2 and 4 blocks an SM
    (2, 2100, (64, 66), 1.0, 3),                                     # exact ties there
]


@pytest.mark.parametrize("dim,n,res,hi,copies", CASES)
@pytest.mark.parametrize("prec", ["fp32", "tf32"])
def test_labels_and_moments(capi, dim, n, res, hi, copies, prec):
    inst = _inst(dim, n, res, hi, copies=copies)
    x, A, w, _ = instance_tensors(inst)
    p = {"fp32": capi.APD_FP32, "tf32": capi.APD_TC_TF32}[prec]
    J, K = inst.grid.num_pixels, oracle.moment_width(dim)
    ws = capi.Workspace(dim, inst.n, J)
    ws.set_pruning(True)
    ref = oracle.assign(inst.grid, inst.x, inst.A, inst.w)
    want = oracle.moments(inst.grid, ref, inst.n)
    lab = torch.full((J,), -1, dtype=torch.int32, device="cuda")
    mom = torch.full((inst.n, K), -3, dtype=torch.int64, device="cuda")
    capi.apd_assign(inst.grid, x, A, w, lab, ws, precision=p)
    assert np.array_equal(host(lab), ref), f"{np.count_nonzero(host(lab) != ref)} labels differ"
    if copies > 1:
        assert ws.last_stats().rescored_fp64 == J
    capi.apd_cell_moments(inst.grid, x, A, w, mom, ws, precision=p)
    np.testing.assert_array_equal(host(mom), want)
    total = np.zeros_like(want)
    r = res[-1]
    for a, b in ((0, 5), (5, r // 2), (r // 2, r)):
        capi.apd_cell_moments_slab(inst.grid, a, b - a, x, A, w, mom, ws, precision=p)
        total += host(mom)
    np.testing.assert_array_equal(total, want)
    assert ws.status() == capi.APD_OK
    b = capi.Batch(dim, [inst.grid, inst.grid], [inst.n, inst.n])
    b.set_pruning(True)
    two = torch.full((2 * inst.n, K), -3, dtype=torch.int64, device="cuda")
    capi.apd_batch_cell_moments(b, torch.cat([x, x]), torch.cat([A, A]), torch.cat([w, w]), two)
    np.testing.assert_array_equal(host(two), np.concatenate([want, want]))


@pytest.mark.parametrize("dim,n,res", [(2, 5000, (100, 96)), (3, 4500, (33, 30, 28))])
def test_solve_takes_the_same_steps(capi, dim, n, res):
    inst = _inst(dim, n, res)
    x, A, _, v = instance_tensors(inst)
    o = capi.solve_opts(eps=1e-9, max_evals=5)
    out = []
    for prune in (False, True):
        ws = capi.Workspace(dim, n, inst.grid.num_pixels)
        ws.set_pruning(prune)
        w = torch.zeros(n, dtype=torch.float64, device="cuda")
        _, info = capi.apd_solve_weights(inst.grid, x, A, torch.zeros_like(w), v, w, ws, o)
        out.append((host(w), info.g, info.evaluations))
    assert out[0][2] == out[1][2]
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
