"""The training step at batches whose samples fall unevenly on the cluster's
eight CTAs (none, one, a partial quad, the full 24), against the oracle's Adam.

Tolerance: Adam's moments after three steps are sums of three gradients (their
squares), each an FP32 sum over the batch with errors of some (64 + 32 + 24)
2^-24 of its terms: 1e-4 of the largest moment, as for the gradient kernel.
"""
import numpy as np
import pytest
import torch

from conftest import balanced_net

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,tail", [(1, 0), (7, 3), (8, 1), (9, 8), (25, 24), (97, 40), (169, 1), (185, 177), (192, 0)])
def test_moments_at_uneven_shares(oracle_mod, tmp_path, batch, tail):
    from oracle import mlp_train
    import paper_2207_08500_gb300 as p
    net = balanced_net(101)
    path = str(tmp_path / "net.bin")
    net.save(path)
    g = p.Neno6(ndim=1, nx=8, weights=path)
    X = synth.mlp_stencils(2000, seed=102)
    rng = np.random.default_rng(103)
    y = rng.integers(0, 16, 2000).astype(np.uint8)
    perm = rng.integers(0, 2000, 2 * batch + (tail or batch)).astype(np.int32)
    q = torch.from_numpy(net.packed().astype(np.float32)).cuda()
    m, v = torch.zeros_like(q), torch.zeros_like(q)
    loss = g.mlp_train(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), torch.from_numpy(perm).cuda(), q, m, v, 0,
                       1e-5, batch=batch)
    assert g.status() == 0
    _, rm, rv, losses = mlp_train.train(net, X, y, perm, batch, 1e-5)
    assert len(losses) == 3 and abs(loss.item() - sum(losses)) <= 1e-5 * sum(losses)
    assert np.abs(m.cpu().numpy() - rm).max() <= 1e-4 * np.abs(rm).max()
    assert np.abs(v.cpu().numpy() - rv).max() <= 1e-4 * np.abs(rv).max()
