"""The adjoint where its tiles end, against the oracle's dual numbers: the
dot-product identity <lambda, J v> = <J^T lambda, v> with v and lambda
supported next to the last faces, on both sides of the sizes at which the
tile changes, and with the mask recomputed against the mask given.

Tolerance: both sides are binary64 sums of at most a few thousand terms of
like size, each with a relative error of some 1e-15 of the largest term;
1e-11 of the sum of magnitudes is far above it and far below any missing or
doubled contribution (one in a few hundred).
"""
import numpy as np
import pytest
import torch

from conftest import balanced_net

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc", [((1, 31), "transmissive"), ((1, 32), "periodic"), ((1, 33), "transmissive"),
                                      ((7, 8), "periodic"), ((8, 7), "transmissive"), ((9, 16), "periodic"),
                                      ((15, 17), "transmissive"), ((399, 383), "periodic"), ((384, 384), "transmissive")])
def test_dot_product_next_to_the_ends(oracle_mod, tmp_path, shape, bc):
    import paper_2207_08500_gb300 as p
    ny, nx = shape
    ndim = 1 if ny == 1 else 2
    net = balanced_net(52)
    path = str(tmp_path / "net.bin")
    net.save(path)
    U = synth.riemann_1d(nx, seed=3) if ndim == 1 else synth.quadrants_2d(nx, ny, seed=3)
    U = synth.noisy(U, seed=4)
    g = p.Neno6(ndim=ndim, nx=nx, ny=ny, bc=(bc, bc), weights=path)
    o = oracle_mod.Oracle(ndim=ndim, nx=nx, ny=ny, bc=(bc, bc), net=net)
    Ud = torch.from_numpy(U).cuda()
    _, mask = g.rhs(Ud, want_mask=True)
    rng = np.random.default_rng(5)
    lam, v = rng.standard_normal(U.shape), rng.standard_normal(U.shape)
    near = np.zeros(U.shape, bool)
    near[:, :, -5:] = near[:, -5:, :] = True
    v = np.where(near, v, 0.0)
    grad = g.rhs_vjp(Ud, torch.from_numpy(lam).cuda(), mask=mask)
    assert torch.equal(grad, g.rhs_vjp(Ud, torch.from_numpy(lam).cuda()))
    grad = grad.cpu().numpy()
    _, Jv = o.jvp(U, v, mask.cpu().numpy())
    a, b = (lam * Jv).sum(), (grad * v).sum()
    assert abs(a - b) <= 1e-11 * max(np.abs(lam * Jv).sum(), np.abs(grad * v).sum())
