"""The pruned scorer (candidate lists over grid regions) where its branches
change: labels and moments equal the FP64 oracle's.

Sizes: one seed; grids of one pixel, one partial tile, one partial region and just
past each; one, two (byte masks), more than eight and more than 48 listed seeds in
a tile, more than one list chunk, and more seeds than a region lists (the tiles
then scan the groups); more than 256 groups; windows that start and end inside
tiles; exact ties of two and of many seeds, whole tiles of them."""
import numpy as np
import pytest

import oracle
from paper_2403_03571_gb300 import synth
from _gpu import host, instance_tensors, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


def _inst(dim, n, res, seed, wscale=0.3, lo=0.0, hi=1.0, cond=0.3):
    g = synth.rng(seed)
    x = lo + (hi - lo) * g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n, cond) if dim == 2 else synth.aniso_3d_lognormal(g, n, cond)
    w = wscale * g.standard_normal(n) * n ** (-2.0 / dim)
    return synth.Instance(synth.Grid(dim, res), x, A, w, np.full(n, 1.0 / n))


def _check(capi, inst, prec="fp32"):
    x, A, w, _ = instance_tensors(inst)
    J, K = inst.grid.num_pixels, oracle.moment_width(inst.grid.dim)
    ws = capi.Workspace(inst.grid.dim, inst.n, J)
    ws.set_pruning(True)
    p = {"fp32": capi.APD_FP32, "tf32": capi.APD_TC_TF32}[prec]
    lab = torch.full((J,), -1, dtype=torch.int32, device="cuda")
    mom = torch.full((inst.n, K), -3, dtype=torch.int64, device="cuda")
    capi.apd_assign(inst.grid, x, A, w, lab, ws, precision=p)
    capi.apd_cell_moments(inst.grid, x, A, w, mom, ws, precision=p)
    assert ws.status() == capi.APD_OK
    ref = oracle.assign(inst.grid, inst.x, inst.A, inst.w)
    assert np.array_equal(host(lab), ref), f"{np.count_nonzero(host(lab) != ref)} labels differ"
    np.testing.assert_array_equal(host(mom), oracle.moments(inst.grid, ref, inst.n))


@pytest.mark.parametrize("dim,n,res", [
    (3, 1, (1, 1, 1)), (3, 2, (7, 9, 8)), (3, 3, (16, 16, 16)), (3, 9, (17, 8, 33)), (3, 200, (31, 18, 9)),
    (3, 40, (64, 5, 3)), (3, 8300, (20, 17, 16)), (3, 1000, (60, 52, 40)),
    (2, 1, (1, 1)), (2, 2, (33, 16)), (2, 5, (64, 64)), (2, 30, (65, 127)), (2, 700, (200, 3)), (2, 400, (130, 250)),
])
def test_labels_and_moments(capi, dim, n, res):
    _check(capi, _inst(dim, n, res, 100 + n))


@pytest.mark.parametrize("dim,n,res", [(3, 40, (16, 16, 16)), (3, 300, (16, 16, 16)), (3, 900, (24, 16, 17)),
                                       (3, 3000, (16, 16, 16)), (2, 500, (64, 64)), (2, 6000, (70, 64))])
@pytest.mark.parametrize("prec", ["fp32", "tf32"])
def test_many_listed_seeds(capi, dim, n, res, prec):
    _check(capi, _inst(dim, n, res, 7 + n, wscale=0.05), prec)


def test_seeds_in_a_corner_and_strong_anisotropy(capi):
    # empty regions far from every seed, and lists much longer than the cells' number
    _check(capi, _inst(3, 2000, (50, 40, 30), 5, lo=0.0, hi=0.12))
    _check(capi, _inst(3, 400, (40, 40, 40), 6, wscale=0.0, cond=1.5))
    _check(capi, _inst(2, 400, (150, 90), 8, cond=1.8))


@pytest.mark.parametrize("dim,res,cuts", [(3, (20, 19, 40), (0, 3, 8, 21, 40)), (2, (100, 150), (0, 5, 64, 70, 150))])
def test_windows_inside_tiles_sum_to_the_grid(capi, dim, res, cuts):
    inst = _inst(dim, 60, res, 11)
    x, A, w, _ = instance_tensors(inst)
    K = oracle.moment_width(dim)
    ws = capi.Workspace(dim, inst.n, inst.grid.num_pixels)
    ws.set_pruning(True)
    total = np.zeros((inst.n, K), dtype=np.int64)
    for a, b in zip(cuts[:-1], cuts[1:]):
        mom = torch.full((inst.n, K), -3, dtype=torch.int64, device="cuda")
        capi.apd_cell_moments_slab(inst.grid, a, b - a, x, A, w, mom, ws)
        total += host(mom)
    assert ws.status() == capi.APD_OK
    ref = oracle.assign(inst.grid, inst.x, inst.A, inst.w)
    np.testing.assert_array_equal(total, oracle.moments(inst.grid, ref, inst.n))


@pytest.mark.parametrize("copies", [2, 5, 60])
def test_ties_of_many_seeds_go_to_the_lowest_index(capi, copies):
    # every seed `copies` times: each pixel ties exactly, in one list chunk and in several
    base = _inst(3, 12, (30, 20, 18), 21)
    idx = np.tile(np.arange(12), copies)
    inst = synth.Instance(base.grid, base.x[idx], base.A[idx], base.w[idx], np.full(len(idx), 1.0 / len(idx)))
    _check(capi, inst)
    x, A, w, _ = instance_tensors(inst)
    ws = capi.Workspace(3, inst.n, inst.grid.num_pixels)
    ws.set_pruning(True)
    lab = torch.empty(inst.grid.num_pixels, dtype=torch.int32, device="cuda")
    capi.apd_assign(inst.grid, x, A, w, lab, ws)
    assert ws.last_stats().rescored_fp64 == inst.grid.num_pixels
    assert int(host(lab).max()) < 12


def test_non_finite_seeds_are_reported(capi):
    inst = _inst(3, 50, (20, 20, 20), 31)
    x, A, w, _ = instance_tensors(inst)
    x[7, 1] = float("nan")
    ws = capi.Workspace(3, inst.n, inst.grid.num_pixels)
    ws.set_pruning(True)
    lab = torch.empty(inst.grid.num_pixels, dtype=torch.int32, device="cuda")
    capi.apd_assign(inst.grid, x, A, w, lab, ws)
    assert ws.status() == capi.APD_ERR_ARG
    assert ws.status() == capi.APD_OK
