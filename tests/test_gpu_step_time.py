"""dt and t of FP64 steps whose tiles are handed out: one CTA alone writes them,
once, whichever has the first tile.

A state repeated periodically has the wave speeds of one period and hence its dt,
bit for bit, and t is the sum of the steps in order, clipped to t_end.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


# 1D: one wave of 31-cell tiles, 127-cell tiles handed out; 2D: one wave of the
# smallest tiles, 7 x 16 and 15 x 16 handed out
@pytest.mark.parametrize("kx,ky", [(1, 0), (220, 0), (1, 1), (8, 8), (16, 10)])
def test_dt_is_that_of_one_period_and_t_their_sum(kx, ky):
    import paper_2207_08500_gb300 as p
    nx, ny = (400, 1) if ky == 0 else (32, 48)
    ndim = 1 if ky == 0 else 2
    U = synth.riemann_1d(nx, seed=81) if ndim == 1 else synth.quadrants_2d(nx, ny, seed=81)
    out = []
    for a, b in ((1, 1), (kx, max(ky, 1))):
        g = p.Neno6(ndim=ndim, nx=nx * a, ny=ny * b, dx=1.0 / nx, dy=1.0 / ny)
        V = torch.from_numpy(np.ascontiguousarray(np.tile(U, (1, b, a)))).cuda()
        t = torch.full((1,), 0.25, dtype=torch.float64, device="cuda")
        dt = torch.zeros(1, dtype=torch.float64, device="cuda")
        dts, ts = [], []
        t_end = 0.0
        for i in range(3):
            if i == 2:
                t_end = ts[-1] + 0.5 * dts[-1]  # the last step is clipped
            dt.fill_(-1.0)
            g.step(V, 0.4, t_end=t_end, t=t, dt=dt)
            dts.append(dt.item())
            ts.append(t.item())
        assert ts[0] == 0.25 + dts[0] and ts[1] == ts[0] + dts[1]
        assert dts[2] == t_end - ts[1] and ts[2] == ts[1] + dts[2]
        assert g.status() == 0
        out.append(dts)
        g.close()
    assert out[0] == out[1]
