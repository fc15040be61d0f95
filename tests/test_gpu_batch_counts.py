"""A batch's per-instance count of pixels settled in FP64.

Every seed is given twice, so at W = 0 each pixel ties exactly and one evaluation settles
all of an instance's pixels in FP64: the count is the instance's pixels, as the
one-instance solver reports it.  There are more regions than resident blocks, and the
blocks' consecutive regions belong to different instances."""
import numpy as np
import pytest

from paper_2403_03571_gb300 import synth
from _gpu import dev, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,sizes", [(2, [(448 + 8 * k, 500 - 9 * k) for k in range(14)]),
                                       (3, [(80 + k, 70 - k, 75) for k in range(7)])])
def test_counts_belong_to_their_instance(dim, sizes):
    require_gpu()
    from paper_2403_03571_gb300 import capi
    insts = []
    for k, res in enumerate(sizes):
        base = synth.make_instance(dim, 12 + k, 8, 40 + k)
        idx = np.repeat(np.arange(base.n), 2)
        insts.append(synth.Instance(synth.Grid(dim, res), base.x[idx], base.A[idx], np.zeros(len(idx)),
                                    0.5 * base.v[idx]))
    x, A, w, v = (dev(a) for a in synth.concat(insts))
    b = capi.Batch(dim, [i.grid for i in insts], [i.n for i in insts])
    b.set_pruning(True)
    o = capi.solve_opts(eps=1e-9, max_evals=1)
    pixels = [i.grid.num_pixels for i in insts]
    for _ in range(5):
        _, infos = capi.apd_batch_solve_weights(b, x, A, w, v, torch.empty_like(w), o)
        assert [i.evaluations for i in infos] == [1] * len(insts)
        assert [i.rescored_fp64 for i in infos] == pixels
    one = insts[0]
    ws = capi.Workspace(dim, one.n, one.grid.num_pixels)
    ws.set_pruning(True)
    zero = torch.zeros(one.n, dtype=torch.float64, device="cuda")
    _, info = capi.apd_solve_weights(one.grid, dev(one.x), dev(one.A), zero, dev(one.v), torch.empty_like(zero), ws, o)
    assert info.rescored_fp64 == pixels[0]
