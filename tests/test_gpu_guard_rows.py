"""The mixed path's FP32 re-evaluation, which takes four flagged rows of a warp
at a time: a row's result may not depend on which rows are flagged with it.

A band above every logit re-evaluates every row (eight full groups per warp);
the narrower ones leave every remainder of four.  All lie above the largest
16-bit logit error seen on 2^20 stencils (1.3 in fp16, 7.5 in bf16), so a row
outside a band has its FP32 sign in 16 bits already and the masks have to agree
bit for bit; and no logit of these states lies within 0.026 of 0, far above
FP32 rounding (some 1e-4 through the network), so they are the oracle's.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,taus", [("fp16", (2.0, 5.0, 17.0, 1e9)), ("bf16", (8.0, 12.0, 23.0, 1e9))])
@pytest.mark.parametrize("nx,ny,bc", [(33, 21, "periodic"), (70, 1, "transmissive"), (57, 30, "transmissive")])
def test_masks_do_not_depend_on_the_rows_flagged_together(oracle_mod, precision, taus, nx, ny, bc):
    import paper_2207_08500_gb300 as p
    U = synth.riemann_1d(nx, seed=23) if ny == 1 else synth.quadrants_2d(nx, ny, seed=28)
    Ud = torch.from_numpy(U).cuda()
    ndim = 1 if ny == 1 else 2
    masks, counts = [], []
    for tau in taus:
        g = p.Neno6(ndim=ndim, nx=nx, ny=ny, bc=(bc, bc), precision=precision, guard_tau=tau)
        d, m = g.rhs(Ud, want_mask=True)
        masks.append(m.cpu().numpy())
        counts.append(g.guard_count())
        assert g.status() == 0
    assert counts == sorted(counts) and counts[-1] == 2 * masks[0].size
    o = oracle_mod.Oracle(ndim=ndim, nx=nx, ny=ny, bc=(bc, bc), net=oracle_mod.Net.load(p.DEFAULT_WEIGHTS))
    assert np.array_equal(masks[-1], o.rhs(U, want_mask=True)[1])
    for m in masks[:-1]:
        assert np.array_equal(m, masks[-1])
