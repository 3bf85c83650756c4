"""The bound with which the FP64 paths' classifier filter certifies a logit's
sign, against an emulation of the filter on the CPU.

The matrix instructions promise their sums in at least single precision, in any
order and with any rounding.  The weakest readings are emulated: additions one
after the other, each cut off at 24 bits, and sums of groups of 4, 8 or 16 products
with the sum before, aligned to the largest addend and cut off below its 24 bits.
The distance to the binary64 network has to stay within the bound for each, on the
trained network and on networks built for the worst: a large addend that many small
ones are added to, and values just above powers of two, whose two binary16 terms
leave the most behind.
"""
import ctypes

import numpy as np
import pytest

from conftest import balanced_net

import synth

W = (6, 64, 32, 16, 8, 4)
# the table's layout in floats: inputs, layer 1, weights of layers 2 to 5, their
# biases, the coefficients of the outputs of layers 2 to 4
IN, W1 = 0, 8
W2 = W1 + 64 * 8
W3 = W2 + 2048
W4 = W3 + 512
W5 = W4 + 128
B = (W5 + 128, W5 + 160, W5 + 176, W5 + 184)
K = (W5 + 192, W5 + 224, W5 + 240)
FLOATS = W5 + 248
U = 2.0 ** -24


def table(net):
    from paper_2207_08500_gb300 import build
    lib = ctypes.CDLL(build.build())
    p = np.ascontiguousarray(net.packed(), dtype=np.float64)
    blob = np.zeros(p.size + FLOATS // 2 + 1)
    f = lib._ZN5neno614build_net_blobERKNS_6NetF64EPv
    f(p.ctypes.data_as(ctypes.c_void_p), blob.ctypes.data_as(ctypes.c_void_p))
    return blob[p.size:].view(np.float32)[:FLOATS]


def weight_terms(T, at, nin, nout):
    """The two binary16 terms [nout][nin] of a layer's weights."""
    tiles = (nout + 7) // 8
    half = T[at:at + (nin + 15) // 16 * tiles * 128].view(np.float16).astype(np.float64)
    hi, lo = np.zeros((nout, nin)), np.zeros((nout, nin))
    for o in range(nout):
        for i in range(nin):
            j = i % 16
            e = 2 * (128 * (i // 16 * tiles + o // 8) + 4 * (4 * (o % 8) + j % 8 // 2) + j // 8) + j % 2
            hi[o, i], lo[o, i] = half[e], half[e + 4]
    return hi, lo


def cut(v, e=None):
    """v cut off (towards 0) at 24 bits of itself or of magnitude 2^e."""
    if e is None:
        _, e = np.frexp(v)
    unit = np.ldexp(1.0, np.maximum(e - 24, -149))
    return np.trunc(v / unit) * unit


def instruction(acc, a, b, group):
    """acc [row][out] + sum over inputs of a [row][in] b [out][in], in groups of
    products aligned with the sum before, or one after the other (group 1)."""
    prod = a[:, None, :] * b[None]
    for i in range(0, prod.shape[2], group):
        if group == 1:
            acc = cut(acc + prod[:, :, i])
            continue
        add = np.concatenate([acc[:, :, None], prod[:, :, i:i + group]], axis=2)
        e = np.frexp(add)[1].max(axis=2, where=add != 0.0, initial=-200)
        acc = cut(cut(add, e[:, :, None]).sum(axis=2))
    return acc


def split(h):
    with np.errstate(over="ignore", invalid="ignore"):
        hi = h.astype(np.float32).astype(np.float16).astype(np.float64)
        return hi, (h - hi).astype(np.float16).astype(np.float64)


def f32(v):
    return v.astype(np.float32).astype(np.float64)


def filtered(net, X, group):
    """Logits (scaled as the table scales them) and the bound, as the kernel
    forms them, and the scales."""
    T = table(net)
    t = T.astype(np.float64)
    # towards-zero conversion, reciprocal off by a unit of the last place
    x = X.astype(np.float32).astype(np.float64)
    x = np.where(np.abs(x) > np.abs(X), np.nextafter(x.astype(np.float32), np.float32(0)), x)
    m = np.maximum(1.0, np.abs(x).max(axis=1, keepdims=True))
    x = f32(x * f32((1 / m) * (1 - 2 * U)))
    err = t[IN] + np.abs(x) @ t[IN + 1:IN + 7]
    w = t[W1:W1 + 512].reshape(64, 8)
    h = np.broadcast_to(w[:, 6], (len(x), 64))
    for j in range(6):
        h = f32(h + x[:, j:j + 1] * w[:, j])
    h = np.maximum(h, 0.0)
    err = err + h @ w[:, 7]
    for l, at in ((1, W2), (2, W3), (3, W4), (4, W5)):
        nin, nout = W[l], W[l + 1]
        whi, wlo = weight_terms(T, at, nin, nout)
        hi, lo = split(h)
        acc = np.broadcast_to(t[B[l - 1]:B[l - 1] + nout], (len(x), nout))
        for k in range(0, nin, 16):
            s = slice(k, k + 16)
            block = np.zeros(acc.shape)
            for a, b in ((lo, whi), (hi, wlo), (hi, whi)):
                block = instruction(block, a[:, s], b[:, s], group)
            acc = f32(acc + block)
        if l < 4:
            h = np.maximum(acc, 0.0)
            err = err + h @ t[K[l - 1]:K[l - 1] + nout]
    b5 = net.layers[-1][1]
    scale = np.where(b5 != 0.0, t[B[3]:B[3] + 4] / np.where(b5 != 0.0, b5, 1.0), np.nan)
    scale[0] = 1.0
    return acc, err, scale


def logits64(net, X):
    h = X / np.maximum(1.0, np.abs(X).max(axis=1, keepdims=True))
    for l, (w, b) in enumerate(net.layers):
        h = h @ w.T + b
        if l < 4:
            h = np.maximum(h, 0.0)
    return h


def worst_net(kind, sign=1.0):
    """Networks whose hidden values hardly depend on the input.  "addends": in
    every sum one product of 1 (0.999 in all but the first) beside products just
    below its last place.  "terms": values just above powers of two."""
    net = balanced_net(71)
    for l in range(5):
        nin, nout = W[l], W[l + 1]
        if kind == "addends":
            one = np.where(np.arange(nout) == 0, 1.0, 0.999)
            w = np.full((nout, nin), sign * 2.0 ** -23 if l else 0.0)
            b = one if l == 0 else np.full(nout, -0.5 if l == 4 else 0.0)
            if l:
                w[:, 0] = one
        else:
            v = 1.0 + 2.0 ** -11 + 2.0 ** -23
            w = np.full((nout, nin), sign * v / nin if l else 0.0)
            b = np.full(nout, v if l == 0 else 2.0 ** (-12 if l == 1 else -6))
        net.layers[l] = (w, b)
    return net


def networks():
    from oracle.weights import Net
    import paper_2207_08500_gb300 as p
    yield "trained", Net.load(p.DEFAULT_WEIGHTS)
    yield "random", balanced_net(72)
    for kind in ("addends", "terms"):
        for sign in (1.0, -1.0):
            yield "%s %+d" % (kind, sign), worst_net(kind, sign)


@pytest.mark.parametrize("group", [1, 4, 8, 16])
def test_no_error_beyond_the_bound(oracle_mod, group):
    X = np.concatenate([synth.mlp_stencils(500, seed=73), 1e-3 * synth.mlp_stencils(100, seed=74)])
    for name, net in networks():
        z, bound, scale = filtered(net, X, group)
        z64 = logits64(net, X) * scale
        ok = np.isfinite(z64)  # a scale that a bias of 0 hides is not compared
        # the scale is read off an FP32 bias: 2 u of the logit
        off = np.abs(z - z64) - 2 * U * np.abs(z64)
        assert ok[:, 0].all() and np.isfinite(bound).all()
        assert (off <= bound[:, None])[ok].all(), (name, (off / bound[:, None])[ok].max())
        if name == "trained":  # and it is of use
            assert (np.abs(z) > bound[:, None]).all(axis=1).mean() > 0.97


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["addends", "terms"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_bits_of_logits_next_to_zero(oracle_mod, tmp_path, kind, sign):
    """The same networks with their logits 1/4 u to 1024 u off 0 on either side:
    the right-hand side's masks are the oracle's, whatever the matrix
    instructions cut off."""
    import torch
    import paper_2207_08500_gb300 as p
    nx = 40
    U = synth.riemann_1d(nx, seed=75)
    net = worst_net(kind, sign)
    w, b = net.layers[-1]
    z = logits64(net, np.zeros((1, 6)))[0]
    off = [s * 2.0 ** e * 2.0 ** -24 for e in range(-2, 11) for s in (1, -1)]
    for i in range(0, len(off), 2):
        for flip in (1.0, -1.0):
            net.layers[-1] = (flip * w, flip * (b - z) + np.array([off[i], off[i + 1], 1.5 * off[i], 1.5 * off[i + 1]]))
            path = str(tmp_path / "net.bin")
            net.save(path)
            g = p.Neno6(ndim=1, nx=nx, bc=("transmissive",) * 2, weights=path)
            m = g.rhs(torch.from_numpy(U).cuda(), want_mask=True)[1].cpu().numpy()
            o = oracle_mod.Oracle(ndim=1, nx=nx, net=net, bc=("transmissive",) * 2)
            assert np.array_equal(m, o.rhs(U, want_mask=True)[1]), (off[i], flip)
            g.close()
