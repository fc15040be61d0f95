"""The unit of length does not matter: coordinates and the box times 2^-k, matrices times
2^2k and the same weights give the same costs of eq. (2.1), bit for bit in FP64, so the
same labels and integer moments, in every form.  k = 22 puts matrices of unit determinant
at determinants of 5e39, beyond FP32."""
import numpy as np
import pytest

import oracle
from oracle import points as op
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    require_gpu()
    from paper_2403_03571_gb300 import capi as c
    return c


def _scaled(dim, n, res, k):
    g = synth.rng(17 + n)
    x = g.random((n, dim))
    A = synth.aniso_2d_lognormal(g, n, 0.3) if dim == 2 else synth.aniso_3d_lognormal(g, n, 0.3)
    w = 0.3 * g.standard_normal(n) * n ** (-2.0 / dim)
    u = 2.0 ** -k
    one = synth.Instance(synth.Grid(dim, res), x, A, w, np.full(n, 1.0 / n))
    grid = synth.Grid(dim, res, (0.0,) * dim, (u,) * dim)
    return one, synth.Instance(grid, u * x, A / u ** 2, w, one.v * u ** dim)


CASES = [(2, 300, (130, 117)), (3, 400, (40, 37, 34))]


@pytest.mark.parametrize("k", [22, -22])
@pytest.mark.parametrize("dim,n,res", CASES)
@pytest.mark.parametrize("prune", [False, True])
@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16"])
def test_assign(capi, dim, n, res, k, prune, prec):
    one, sc = _scaled(dim, n, res, k)
    ws = capi.Workspace(dim, n, one.grid.num_pixels)
    ws.set_pruning(prune)
    p = {"fp32": capi.APD_FP32, "tf32": capi.APD_TC_TF32, "bf16": capi.APD_TC_BF16}[prec]
    lab = torch.full((one.grid.num_pixels,), -1, dtype=torch.int32, device="cuda")
    mom = torch.full((n, oracle.moment_width(dim)), -1, dtype=torch.int64, device="cuda")
    capi.apd_assign(sc.grid, dev(sc.x), dev(sc.A), dev(sc.w), lab, ws, precision=p)
    capi.apd_cell_moments(sc.grid, dev(sc.x), dev(sc.A), dev(sc.w), mom, ws, precision=p)
    assert ws.status() == capi.APD_OK
    ref = oracle.assign(one.grid, one.x, one.A, one.w)
    assert np.array_equal(host(lab), ref), f"{np.count_nonzero(host(lab) != ref)} labels differ"
    assert np.array_equal(host(mom), oracle.moments(one.grid, ref, n))


@pytest.mark.parametrize("k", [22, -22])
@pytest.mark.parametrize("dim,n,res", CASES)
def test_masked_batch_and_points(capi, dim, n, res, k):
    one, sc = _scaled(dim, n, res, k)
    x, A, w = dev(sc.x), dev(sc.A), dev(sc.w)
    ws = capi.Workspace(dim, n, one.grid.num_pixels)
    ws.set_pruning(True)
    out = []
    for i in (one, sc):
        lab = torch.full((one.grid.num_pixels,), -1, dtype=torch.int32, device="cuda")
        mom = torch.full((n, oracle.moment_width(dim)), -1, dtype=torch.int64, device="cuda")
        capi.apd_masked_moments(i.grid, 2, dev(i.x), dev(i.A), dev(i.w), mom, lab, ws)
        assert ws.status() == capi.APD_OK
        out.append((host(lab), host(mom)))
    ref = oracle.assign(one.grid, one.x, one.A, one.w)
    assert np.array_equal(out[1][0], ref)
    assert np.array_equal(out[0][1], out[1][1])
    for prune in (False, True):
        b = capi.Batch(dim, [sc.grid, sc.grid], [n, n])
        b.set_pruning(prune)
        mom = torch.full((2 * n, oracle.moment_width(dim)), -1, dtype=torch.int64, device="cuda")
        capi.apd_batch_cell_moments(b, torch.cat([x, x]), torch.cat([A, A]), torch.cat([w, w]), mom)
        want = oracle.moments(one.grid, ref, n)
        assert np.array_equal(host(mom), np.concatenate([want, want]))
    for m in (n, 8):  # the tiled and the direct form
        y = np.random.default_rng(n + m).random((4000, dim))
        lab = torch.full((4000,), -1, dtype=torch.int32, device="cuda")
        mom = torch.empty((m, op.moment_width(dim)), dtype=torch.float64, device="cuda")
        mass = torch.full((4000,), 1.0, dtype=torch.float64, device="cuda")
        capi.apd_points_moments(dev(2.0 ** -k * y), mass, x[:m].contiguous(), A[:m].contiguous(), w[:m].contiguous(), mom,
                                ws, labels=lab)
        assert ws.status() == capi.APD_OK
        assert np.array_equal(host(lab), op.assign(y, one.x[:m], one.A[:m], one.w[:m]))
