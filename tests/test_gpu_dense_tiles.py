"""The dense scorer's groups of eight seeds, its chunks of 256 held three (3D) or four (2D)
at a time, and both tile sizes: labels and moments are integers and equal the FP64 oracle's."""
import numpy as np
import pytest

import oracle
from paper_2403_03571_gb300 import synth
from _gpu import host, instance_tensors, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,res", [
    # small tiles (8^3, 32 x 16): below, at and just past a tile; one group of eight and one more
    (3, 1, (1, 1, 1)), (3, 7, (8, 8, 8)), (3, 8, (9, 7, 17)), (3, 9, (16, 33, 8)), (2, 8, (32, 16)), (2, 17, (33, 65)),
    # chunk edges
    (3, 255, (20, 20, 20)), (2, 256, (100, 70)), (3, 257, (20, 19, 18)), (3, 769, (24, 20, 17)), (2, 1025, (90, 110)),
    # large tiles: 80 or more of them, ragged; held chunks: all, one past, two rounds
    (3, 33, (79, 66, 70)), (3, 768, (70, 79, 65)), (3, 769, (65, 70, 79)), (3, 1600, (79, 65, 70)),
    (2, 30, (577, 600)), (2, 1024, (600, 577)), (2, 1025, (577, 590)), (2, 2100, (590, 577)),
])
@pytest.mark.parametrize("ties", [False, True])
def test_dense_labels_and_moments(dim, n, res, ties):
    require_gpu()
    from paper_2403_03571_gb300 import capi
    g = synth.rng(31 + n)
    x = g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n, 0.3) if dim == 2 else synth.aniso_3d_lognormal(g, n, 0.3)
    w = 0.2 * g.standard_normal(n) * n ** (-2.0 / dim)
    if ties and n > 1:  # every other seed again: exact ties, the lower index wins
        x[1::2], A[1::2], w[1::2] = x[:n - 1:2][:n // 2], A[:n - 1:2][:n // 2], w[:n - 1:2][:n // 2]
    inst = synth.Instance(synth.Grid(dim, res), x, A, w, np.full(n, 1.0 / n))
    xd, Ad, wd, _ = instance_tensors(inst)
    ws = capi.Workspace(dim, n, inst.grid.num_pixels)
    ws.set_pruning(False)
    lab = torch.full((inst.grid.num_pixels,), -1, dtype=torch.int32, device="cuda")
    mom = torch.full((n, oracle.moment_width(dim)), -3, dtype=torch.int64, device="cuda")
    capi.apd_assign(inst.grid, xd, Ad, wd, lab, ws)
    capi.apd_cell_moments(inst.grid, xd, Ad, wd, mom, ws)
    assert ws.status() == capi.APD_OK
    ref = oracle.assign(inst.grid, x, A, w)
    assert np.array_equal(host(lab), ref), f"{np.count_nonzero(host(lab) != ref)} labels differ"
    np.testing.assert_array_equal(host(mom), oracle.moments(inst.grid, ref, n))
