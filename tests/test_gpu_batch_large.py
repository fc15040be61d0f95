"""Batched solves on both sides of the solver kernel's and the records' size limits (2048
seeds kept in registers, 4096 sorted, 8192 groups handled a lane each) and with pruning
switched on and off between calls, against the one-instance solver.

Tolerance: both take the same steps from integer moments; their direction sums differ in
association, by at most ~n * 1.1e-16 = 1e-12 relative a direction, and three evaluations
apply two of them: 1e-9 leaves a factor of 500 for their conditioning."""
import numpy as np
import pytest

from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("evals", [1, 3])
def test_large_instances_follow_the_single_solver(evals):
    require_gpu()
    from paper_2403_03571_gb300 import capi
    specs = [(2047, 128), (2048, 128), (2049, 128), (4097, 160), (8193, 200), (1, 8), (33, 24)]
    insts = [synth.make_instance(2, n, m, 900 + n) for n, m in specs]
    x, A, _, v = (dev(a) for a in synth.concat(insts))
    b = capi.Batch(2, [i.grid for i in insts], [i.n for i in insts])
    o = capi.solve_opts(eps=1e-9, max_evals=evals)
    out = {}
    for prune in (False, True, False):  # the records and the iteration's graph follow the switch
        b.set_pruning(prune)
        w = torch.zeros_like(v)
        _, infos = capi.apd_batch_solve_weights(b, x, A, torch.zeros_like(v), v, w, o)
        out.setdefault(prune, (host(w), [i.g for i in infos], [i.evaluations for i in infos]))
    assert np.array_equal(out[False][0], out[True][0])  # the same labels, moments and steps
    off = 0
    for k, inst in enumerate(insts):
        ws = capi.Workspace(2, inst.n, inst.grid.num_pixels)
        ws.set_pruning(True)
        w1 = torch.zeros(inst.n, dtype=torch.float64, device="cuda")
        _, info = capi.apd_solve_weights(inst.grid, dev(inst.x), dev(inst.A), torch.zeros_like(w1), dev(inst.v), w1,
                                         ws, o)
        got = out[True][0][off:off + inst.n]
        off += inst.n
        assert out[True][2][k] == info.evaluations
        assert out[True][1][k] == pytest.approx(info.g, rel=1e-9, abs=1e-15)
        scale = max(np.abs(host(w1)).max(), 1e-30)
        assert np.abs(got - host(w1)).max() <= 1e-9 * scale
