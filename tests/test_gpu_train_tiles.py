"""The network kernels take 32 samples per block and at most 608 blocks keep a gradient
partial: batches at the edges of a tile and of the partials, against the FP64 oracle.

Tolerance: a 64-term FP32 chain errs by at most ~64 * 6e-8 of the terms' magnitudes, three
layers forward and back by ~2.4e-5; 1e-4 of the largest entry (1e-3 relative) is four times that."""
import numpy as np
import pytest

from oracle import warmstart as ow
from paper_2403_03571_gb300 import synth
from _gpu import dev, host, require_gpu, torch

pytestmark = pytest.mark.gpu


def _net(dim):
    require_gpu()
    from paper_2403_03571_gb300 import capi
    g = np.random.Generator(np.random.PCG64(40 + dim))
    F, P = ow.n_features(dim), ow.n_params(dim)
    params = (g.normal(0, 0.15, P)).astype(np.float32)
    norm = np.concatenate([g.normal(0, 0.5, F), np.exp(g.normal(0, 0.3, F))]).astype(np.float32)
    return capi.WarmStart(dim, params, norm), params.astype(np.float64), norm.astype(np.float64), g


@pytest.mark.parametrize("dim,B", [(2, 1), (3, 31), (2, 32), (3, 33), (2, 608 * 32), (3, 608 * 32 + 1),
                                   (2, 2 * 608 * 32 + 33)])
def test_gradient_at_tile_edges(dim, B):
    net, params, norm, g = _net(dim)
    feats = g.normal(0.3, 1.5, (B + 3, ow.n_features(dim))).astype(np.float32)
    targets = g.normal(0, 1, B + 3).astype(np.float32)
    idx = g.permutation(B + 3)[:B].astype(np.int32)
    grad = torch.zeros(ow.n_params(dim), dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    net.train_step(dev(idx), dev(feats), dev(targets), 0.0, grad_out=grad, loss_out=loss)
    L, ref = ow.loss_grad(params, norm, feats[idx].astype(np.float64), targets[idx].astype(np.float64), dim)
    assert float(host(loss)[0]) == pytest.approx(L * B, rel=1e-4)
    np.testing.assert_allclose(host(grad), ref, rtol=1e-3, atol=1e-4 * np.abs(ref).max())


@pytest.mark.parametrize("dim,n", [(2, 1), (3, 31), (2, 33), (3, 96)])
def test_prediction_at_tile_edges(dim, n):
    net, params, norm, g = _net(dim)
    feats = g.normal(0.3, 1.5, (n, ow.n_features(dim))).astype(np.float32)
    grid = synth.Grid(dim, (8,) * dim)
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    net.predict([n], [grid], dev(feats), out)
    ref = ow.predict(params, norm, feats.astype(np.float64), n, grid.measure, dim)
    np.testing.assert_allclose(host(out), ref, rtol=1e-4, atol=2e-5 * np.abs(ref).max())
