"""Bulk classification with its tiles handed out, where a CTA's warps drift apart.

Every thread of a CTA goes on to the tile that one thread asked for.  With the
outputs in mapped host memory the warps leave a tile far apart, as their stores
are slow and uneven, and a warp that took its number from a word already
written for the round after would leave rows out or put them under another
tile's index: every row has to be that of the same call on less than the
12 x 1216 tiles from which tiles are handed out.
"""
import ctypes

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12 * 1216 * 128 - 127, 2500017])
def test_rows_are_their_own_when_warps_drift_apart(n):
    import paper_2207_08500_gb300 as p
    g = p.Neno6(ndim=1, nx=64, precision="fp16")
    base = torch.from_numpy(synth.mlp_stencils(100003, seed=47)).cuda()
    X = base.repeat((n + 100002) // 100003, 1)[:n].contiguous()
    half = n // 2  # dealt out beforehand
    parts = [g.classify(x, want_logits=True) for x in (X[:half], X[half:])]
    e1, z1 = (torch.cat([q[i] for q in parts]).cpu() for i in range(2))
    eta = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    z = torch.empty((n, 4), dtype=torch.float64, pin_memory=True)
    lib = p.load_library()
    at = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    for with_logits in (True, False, True):
        eta.fill_(255)
        z.fill_(float("nan"))
        torch.cuda.synchronize()
        assert lib.neno6_classify(g._h, at(X), n, at(eta), at(z) if with_logits else None, None) == 0
        torch.cuda.synchronize()
        assert torch.equal(eta, e1)
        if with_logits:
            assert torch.equal(z, z1)
    assert g.status() == 0
