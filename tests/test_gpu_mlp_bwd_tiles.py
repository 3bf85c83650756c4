"""The FP32 loss gradient where its 128-sample tiles and its CTAs end, against
the FP64 oracle gradient.

Tolerance: a gradient entry is a sum of n products with relative errors of
some (64 + 32) 2^-24 from the layers, summed in FP32 in chains of at most a
few thousand terms: 2e-4 of the largest entry, as for the whole-size check.
"""
import numpy as np
import pytest
import torch

from conftest import balanced_net

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 17, 128, 129, 256, 152 * 128 - 1, 152 * 128 + 1, 2 * 152 * 128 + 77])
def test_mlp_bwd_tile_edges(tmp_path, n):
    from oracle import mlp_grad
    import paper_2207_08500_gb300 as p
    net = balanced_net(75)
    path = str(tmp_path / "net.bin")
    net.save(path)
    X = synth.mlp_stencils(n, seed=76)
    y = np.random.default_rng(77).integers(0, 16, n).astype(np.uint8)
    g = p.Neno6(ndim=1, nx=8, weights=path)
    grad, loss = g.mlp_bwd(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    again, _ = g.mlp_bwd(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    assert torch.equal(grad, again)
    ref = mlp_grad.grad(net, X, y)
    assert np.abs(grad.cpu().numpy() - ref).max() <= 2e-4 * np.abs(ref).max()
    assert abs(float(loss) - mlp_grad.loss(net, X, y)) <= 2e-5 * abs(mlp_grad.loss(net, X, y))
