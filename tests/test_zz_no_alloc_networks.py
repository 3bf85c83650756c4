"""neno6_step_noalloc with another network at every call, on grids whose kernels
may start before the one ahead of them has finished.

Each call lays its network out in the shared static array on the stream and the
kernels of the same call read it from there: calls that follow one another
without a synchronisation must each use their own.  The kernels are those of
neno6_step, so the states agree bit for bit.  Collected last, as it uses the
static array.
"""
import ctypes

import numpy as np
import pytest
import torch

from conftest import balanced_net

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 64), (1, 2300), (16, 24), (40, 48)])
def test_each_call_uses_its_own_network(tmp_path, shape):
    import paper_2207_08500_gb300 as p
    ny, nx = shape
    ndim = 1 if ny == 1 else 2
    U0 = np.ascontiguousarray(synth.smooth_2d(nx, max(ny, 2), seed=61)[:, :ny])
    if ndim == 1:  # density, momentum, energy of the row at rest across it
        U0 = np.stack([U0[0], U0[1], U0[3] - 0.5 * U0[2] ** 2 / U0[0]])
    nets, handles = [], []
    for seed in (62, 63):
        net = balanced_net(seed)
        path = str(tmp_path / ("net%d.bin" % seed))
        net.save(path)
        nets.append(np.ascontiguousarray(net.packed(), dtype=np.float64))
        handles.append(p.Neno6(ndim=ndim, nx=nx, ny=ny, weights=path))
    c = p._Config()
    c.ndim, c.nx, c.ny = ndim, nx, ny
    c.dx, c.dy, c.gamma = 1.0 / nx, 1.0 / ny, 1.4
    c.bc[0] = c.bc[1] = p.BC["periodic"]
    c.precision, c.linear_weights, c.mask_mode = 0, 0, 0
    calls = 24
    U = torch.from_numpy(U0).cuda()
    V, W = U.clone(), U.clone()
    for i in range(calls):
        handles[i % 2].step(U, 0.3)
        handles[0].step(W, 0.3)
    torch.cuda.synchronize()
    lib = p.load_library()
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for i in range(calls):
        w = nets[i % 2]
        assert lib.neno6_step_noalloc(ctypes.byref(c), w.ctypes.data_as(ctypes.c_void_p), w.size,
                                      ctypes.c_void_p(V.data_ptr()), 0.3, 0.0, None, None, None, stream) == 0
    torch.cuda.synchronize()
    assert torch.isfinite(U).all() and not torch.equal(U, W)  # the networks differ on this state
    assert torch.equal(U, V)
