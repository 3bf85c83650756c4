"""Faces between physical cells whose Roe average has no sound speed.

At extreme Mach numbers the average of two cells with positive pressure can round
to c^2 <= 0.  Its eigenvectors are then infinite or NaN, and the right-hand side
is NaN next to the face, as the oracle's is, with the status bit set; every other
cell is the oracle's bit for bit.
"""
import numpy as np
import pytest
import torch

from conftest import balanced_net

pytestmark = pytest.mark.gpu


def state(ndim, n, seed):
    """Velocity 2^20 up to rounding, pressures of one to three units of the
    energy's last place."""
    rng = np.random.default_rng(seed)
    rho = rng.uniform(0.5, 2.0, n)
    m = rho * (2.0 ** 20 * (1.0 + 1e-12 * rng.standard_normal(n)))
    u = m / rho
    E = 0.5 * (rho * (u * u))
    E = E + rng.integers(1, 4, n) * np.spacing(E)
    assert (E - 0.5 * (rho * (u * u)) > 0.0).all()
    if ndim == 1:
        return np.stack([rho, m, E])[:, None, :].copy()
    return np.repeat(np.stack([rho, m, 0.0 * m, E])[:, None, :], 9, axis=1).copy()


@pytest.mark.parametrize("ndim,n", [(1, 16), (1, 20000), (2, 16), (2, 400), (2, 4000)])
def test_no_sound_speed_is_nan_next_to_the_face(oracle_mod, tmp_path, ndim, n):
    import paper_2207_08500_gb300 as p
    net = balanced_net(33)
    path = str(tmp_path / "net.bin")
    net.save(path)
    for seed in (0, 3, 6):
        U = state(ndim, n, seed)
        if ndim == 2 and n >= 400:
            U = np.repeat(U, 12, axis=1).copy()
        ny = U.shape[1]
        kw = dict(ndim=ndim, nx=n, ny=ny, bc=("transmissive", "transmissive"))
        g = p.Neno6(weights=path, **kw)
        d = g.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
        ref = oracle_mod.Oracle(net=net, **kw).rhs(U)
        assert g.status() == (2 if np.isnan(ref).any() else 0)
        assert np.array_equal(d, ref, equal_nan=True), (seed, np.isnan(ref).sum(), np.isnan(d).sum())
        g.close()
