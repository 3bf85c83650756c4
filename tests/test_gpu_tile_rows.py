"""The tensor-core classifier and gradient fetch a tile of stencils ahead by bulk
copies where X is 16-byte aligned: equal, bit for bit, to the same stencils at an
address that is only 8-byte aligned (plain loads), at the ends of tiles and of the
persistent grid, with values whose conversion to FP32 is not a normal number.
"""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def both(n, seed):
    X = torch.from_numpy(synth.mlp_stencils(max(n, 2), seed=seed)[:n].copy())
    X[::7, 2] = 0.0
    X[::11, 3] = -1e-41   # subnormal in FP32
    X[::13, 1] = 1e-60    # below the FP32 range
    X[5::17, 0] = 3e38
    X[6::19, 5] = -0.0
    buf = torch.empty(6 * n + 2, dtype=torch.float64, device="cuda")
    b = 1 - buf.data_ptr() % 16 // 8
    A = X.cuda()
    B = buf[b:b + 6 * n].view(n, 6)
    B.copy_(A)
    assert A.data_ptr() % 16 == 0 and B.data_ptr() % 16 == 8
    return A, B


@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 1000, 128 * 1216 + 1, 128 * 1216 * 2 + 77])
def test_aligned_rows_equal_unaligned_ones(precision, n):
    import paper_2207_08500_gb300 as p
    A, B = both(n, 5)
    g = p.Neno6(ndim=1, nx=8, precision=precision)
    ea, za = g.classify(A, want_logits=True)
    eb, zb = g.classify(B, want_logits=True)
    assert torch.equal(ea, eb) and torch.equal(za, zb)
    y = (torch.arange(n, device="cuda") % 16).to(torch.uint8)
    ga, la = g.mlp_bwd(A, y)
    gb, lb = g.mlp_bwd(B, y)
    assert torch.equal(ga, gb) and torch.equal(la, lb)
    assert g.status() == 0
