"""Pruned passes that the region scorer does not take: more seeds than it lists (16384), and
grids of hardly more pixels than seeds.  FP32, and TF32 and BF16 with matrices mild enough
for the tensor-core lists; labels, moments and a batch with such an instance equal the FP64
oracle's."""
import numpy as np
import pytest

import oracle
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


def _inst(dim, n, res, sigma, copies=1):
    g = synth.rng(n + dim)
    x = g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n, sigma) if dim == 2 else synth.aniso_3d_lognormal(g, n, sigma)
    w = 0.3 * g.standard_normal(n) * n ** (-2.0 / dim)
    idx = np.tile(np.arange(n), copies)
    return synth.Instance(synth.Grid(dim, res), x[idx], A[idx], w[idx], np.full(len(idx), 1.0 / len(idx)))


@pytest.mark.parametrize("dim,n,res,copies", [(3, 16385, (34, 30, 33), 1), (2, 16900, (130, 127), 1),
                                              (3, 4097, (20, 17, 28), 1), (2, 4300, (100, 101), 1),
                                              (3, 9000, (40, 41, 42), 1), (2, 8450, (64, 66), 2)])
@pytest.mark.parametrize("prec,sigma", [("fp32", 0.3), ("tf32", 0.08), ("bf16", 0.08)])
def test_labels_and_moments(capi, dim, n, res, copies, prec, sigma):
    inst = _inst(dim, n, res, sigma, copies)
    p = {"fp32": capi.APD_FP32, "tf32": capi.APD_TC_TF32, "bf16": capi.APD_TC_BF16}[prec]
    x, A, w = dev(inst.x), dev(inst.A), dev(inst.w)
    ws = capi.Workspace(dim, inst.n, inst.grid.num_pixels)
    ws.set_pruning(True)
    lab = torch.full((inst.grid.num_pixels,), -1, dtype=torch.int32, device="cuda")
    mom = torch.full((inst.n, oracle.moment_width(dim)), -3, dtype=torch.int64, device="cuda")
    capi.apd_assign(inst.grid, x, A, w, lab, ws, precision=p)
    capi.apd_cell_moments(inst.grid, x, A, w, mom, ws, precision=p)
    assert ws.status() == capi.APD_OK
    ref = oracle.assign(inst.grid, inst.x, inst.A, inst.w)
    assert np.array_equal(host(lab), ref), f"{np.count_nonzero(host(lab) != ref)} labels differ"
    np.testing.assert_array_equal(host(mom), oracle.moments(inst.grid, ref, inst.n))


@pytest.mark.parametrize("dim,specs", [(2, [(16500, (90, 80)), (40, (70, 64))]), (3, [(30, (20, 21, 22)), (16600, (24, 20, 22))])])
def test_batch_with_one_such_instance(capi, dim, specs):
    insts = [_inst(dim, n, res, 0.3) for n, res in specs]
    x, A, w, _ = (dev(a) for a in synth.concat(insts))
    b = capi.Batch(dim, [i.grid for i in insts], [i.n for i in insts])
    want = np.concatenate([oracle.moments(i.grid, oracle.assign(i.grid, i.x, i.A, i.w), i.n) for i in insts])
    for prune in (True, False):
        b.set_pruning(prune)
        mom = torch.full((x.shape[0], oracle.moment_width(dim)), -3, dtype=torch.int64, device="cuda")
        capi.apd_batch_cell_moments(b, x, A, w, mom)
        np.testing.assert_array_equal(host(mom), want)
