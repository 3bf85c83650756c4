"""The face blocks of the mixed kernel and the tiles of the FP64 one, handed out to
the running CTAs as they finish.

A state tiled periodically from whole face blocks (64 x 48 cells) gives every
block the stencils, the reference state and hence the bits of its counterpart
in the small grid, so dU/dt and the masks of the large grid are those of the
small one, repeated: a block left out, taken twice or misplaced shows.  Sizes on
both sides of the 1216 blocks that run at once, and far above; the FP64 result
does not depend on the tile at all.
"""
import os

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,mode", [("fp16", "mlp"), ("bf16", "mlp"), ("fp16", "smooth"), ("fp64", "mlp")])
@pytest.mark.parametrize("kx,ky", [(3, 3), (4, 3), (7, 5), (16, 16)])
def test_a_tiled_state_gives_a_tiled_result(precision, mode, kx, ky):
    import paper_2207_08500_gb300 as p
    nx, ny = 64, 48
    U = synth.noisy(synth.quadrants_2d(nx, ny, seed=41), 42)
    out = []
    for a, b in ((1, 1), (kx, ky)):
        g = p.Neno6(ndim=2, nx=nx * a, ny=ny * b, dx=1.0 / nx, dy=1.0 / ny, precision=precision, mask_mode=mode)
        V = torch.from_numpy(np.ascontiguousarray(np.tile(U, (1, b, a)))).cuda()
        d = torch.full_like(V, float("nan"))
        for _ in range(3):
            d.copy_(g.rhs(V))
        m = g.rhs(V, want_mask=True)[1].cpu().numpy() if mode == "mlp" else None
        assert g.status() == 0
        out.append((d.cpu().numpy(), m, nx * a, ny * b))
    (d1, m1, _, _), (d2, m2, NX, NY) = out
    assert np.array_equal(np.tile(d1, (1, ky, kx)), d2)
    if m1 is not None:
        def split(m, w, h):  # x faces (4, h, w + 1), then y faces (4, h + 1, w)
            n = 4 * h * (w + 1)
            return m.reshape(-1)[:n].reshape(4, h, w + 1)[:, :, :-1], m.reshape(-1)[n:].reshape(4, h + 1, w)[:, :-1]
        for s, l in zip(split(m1, nx, ny), split(m2, NX, NY)):
            assert np.array_equal(np.tile(s, (1, ky, kx)), l)


@pytest.mark.parametrize("width", ["paper", "narrow"])
@pytest.mark.parametrize("n", [12 * 1216 * 128 - 128, 12 * 1216 * 128 - 127, 12 * 1216 * 128 + 1, 2500017])
def test_classify_repeats_a_repeated_input(width, n):
    """Both sides of the 12 x 1216 tiles of 128 rows from which tiles are handed
    out: rows repeated with a period that no tile divides give repeated results."""
    import paper_2207_08500_gb300 as p
    weights = p.DEFAULT_WEIGHTS
    if width == "narrow":
        weights = os.path.join(os.path.dirname(weights), "neno6_mlp_6x32x32x32x4.bin")
    g = p.Neno6(ndim=1, nx=64, precision="fp16", weights=weights)
    base = torch.from_numpy(synth.mlp_stencils(1009, seed=43)).cuda()
    X = base.repeat((n + 1008) // 1009, 1)[:n].contiguous()
    e1, z1 = g.classify(base, want_logits=True)
    e2, z2 = g.classify(X, want_logits=True)
    k = torch.arange(n, device="cuda") % 1009
    assert torch.equal(e2, e1[k]) and torch.equal(z2, z1[k])
    assert torch.equal(g.classify(X), e2)
    assert g.status() == 0
