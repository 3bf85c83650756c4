"""The FP64 right-hand side where its certified FP32 classifier cannot decide
and where its tiles end, against the oracle bit for bit.

The filter may only ever pass on the binary64 network's own bits, so the
tolerance is zero throughout: masks and dU/dt equal the oracle's exactly.
"""
import numpy as np
import pytest
import torch

from conftest import balanced_net

import synth

pytestmark = pytest.mark.gpu


def check(tmp_path, net, U, bc="periodic"):
    import oracle
    import paper_2207_08500_gb300 as p
    path = str(tmp_path / "net.bin")
    net.save(path)
    ndim, ny, nx = (1, 1, U.shape[2]) if U.shape[0] == 3 else (2, U.shape[1], U.shape[2])
    g = p.Neno6(ndim=ndim, nx=nx, ny=ny, bc=(bc, bc), weights=path)
    d, m = g.rhs(torch.from_numpy(U).cuda(), want_mask=True)
    o = oracle.Oracle(ndim=ndim, nx=nx, ny=ny, net=net, bc=(bc, bc))
    d_o, m_o = o.rhs(U, want_mask=True)
    assert np.array_equal(m.cpu().numpy(), m_o)
    assert np.array_equal(d.cpu().numpy(), d_o)
    return m_o


def test_logits_within_rounding_of_zero(oracle_mod, tmp_path):
    """Output biases that put one field's logits within ~1e-7 of 0 on an
    almost uniform state: rows by the thousand that FP32 cannot decide, a few
    per warp and whole warps of them."""
    rng = np.random.default_rng(3)
    nx, ny = 49, 35
    one = np.ones((ny, nx))
    U = synth.prim_to_cons(one, 0.3 * one, -0.2 * one, one)
    U = U * (1.0 + 1e-8 * rng.standard_normal(U.shape))
    net = balanced_net(31)
    # the entropy field's "+" side of x faces: L_1 U, L_1 F of the uniform state
    c2, q = 1.4, 0.13
    b1 = 0.4 / c2
    L = np.array([1 - 0.5 * b1 * q, b1 * 0.3, -b1 * 0.2, -b1])
    E = U[3].mean()
    s = 0.5 * (L @ [0.3, 1.09, -0.06, (E + 1) * 0.3] + 0.3 * (L @ [1, 0.3, -0.2, E]))
    o = oracle_mod.Oracle(ndim=1, nx=8, net=net)
    _, z = o.classify(np.full((1, 6), s))
    W, b = net.layers[-1]
    net.layers[-1] = (W, b - z[0])
    m = check(tmp_path, net, U)
    assert len(np.unique(m)) > 2  # both signs occur


@pytest.mark.parametrize("layer,scale", [(-1, 0.0), (2, 1e30), (2, 1e60), (1, 3e4), (2, 3e5), (0, 2e5), (3, 1e-6),
                                         (1, 1e-7)])
def test_networks_at_the_ends_of_the_number_ranges(oracle_mod, tmp_path, layer, scale):
    """All logits 0 (nothing is certified); weights or hidden values beyond the
    FP32 and the binary16 range, and below the binary16 normal range."""
    net = balanced_net(32)
    W, b = net.layers[layer]
    net.layers[layer] = (W * scale, b * scale)
    check(tmp_path, net, synth.quadrants_2d(21, 18, seed=4))


@pytest.mark.parametrize("kind", ["tiny momentum", "huge", "subnormal momentum"])
@pytest.mark.parametrize("nx,ny", [(20, 17), (70, 1)])
def test_tiles_with_extreme_values(oracle_mod, tmp_path, kind, nx, ny):
    """Values for which halving the eigenvector rows would not be exact."""
    U = synth.riemann_1d(nx, seed=6) if ny == 1 else synth.quadrants_2d(nx, ny, seed=6)
    if kind == "huge":
        U = U * 2.0 ** 300
    else:
        U[1] = (1e-290 if kind == "tiny momentum" else 3e-310) * np.sign(U[1])
        if ny > 1:
            U[2] = 2.5e-308 * np.sign(U[2])
    check(tmp_path, balanced_net(33), U, bc="transmissive")


# the last four lie on both sides of the sizes at which the tile changes
@pytest.mark.parametrize("nx,ny", [(1, 1), (15, 16), (16, 15), (17, 33), (48, 16), (31, 3), (3, 31), (130, 65),
                                   (133, 48), (134, 48), (168, 152), (169, 152)])
@pytest.mark.parametrize("bc", ["periodic", "transmissive"])
def test_tile_edges_2d(oracle_mod, tmp_path, nx, ny, bc):
    check(tmp_path, balanced_net(34), synth.noisy(synth.quadrants_2d(nx, ny, seed=7), 8), bc)


@pytest.mark.parametrize("nx", [1, 5, 30, 31, 32, 63, 127, 383, 18848, 18849])
def test_tile_edges_1d(oracle_mod, tmp_path, nx):
    check(tmp_path, balanced_net(35), synth.riemann_1d(nx, seed=9), "transmissive")


@pytest.mark.parametrize("nx,ny", [(15 * 61 - 4, 16 * 60 - 7), (15 * 24 - 4, 16 * 38 - 7), (15 * 23 - 4, 16 * 38 - 7)])
def test_large_grid_tile(oracle_mod, tmp_path, nx, ny):
    """The tile of large grids (from 912 tiles of 15 x 16) on ragged grids, and
    the next smaller one just below: equal to the oracle on a band of rows cut
    out with its halo."""
    import oracle
    import paper_2207_08500_gb300 as p
    r0, r1 = 300, 340
    U = synth.noisy(synth.quadrants_2d(nx, ny, seed=10), 11)
    net = balanced_net(36)
    path = str(tmp_path / "net.bin")
    net.save(path)
    g = p.Neno6(ndim=2, nx=nx, ny=ny, weights=path)
    d = g.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    cut = np.ascontiguousarray(U[:, r0 - 3:r1 + 3])
    o = oracle.Oracle(ndim=2, nx=nx, ny=r1 - r0 + 6, net=net, dx=1.0 / nx, dy=1.0 / ny)
    assert np.array_equal(d[:, r0:r1], o.rhs(cut)[:, 3:-3])
