"""Blocks whose rows or addresses fit no vector access: the corner turns, the
8-bit plane split and the packet turn against the oracle / the plain
permutation (whole numbers, so equality)."""
import numpy as np
import pytest

import oracle
from paper_1904_07778_gb300 import synth

pytestmark = pytest.mark.gpu

# inputs, channels, spectra around the turn's 256 x 128 tiles and 32-byte pieces
SHAPES = [(1, 1, 1), (3, 5, 31), (5, 3, 33), (13, 10, 255), (100, 2, 257), (37, 7, 513), (33, 31, 96)]


def _push(N, C, T, bits, layout, shift, seed=3):
    """Visibilities of a device block that starts `shift` bytes past an aligned address."""
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    b = synth.random_bytes(seed, N * C * T * bits // 4)
    if bits == 8:
        b[b == 0x80] = 0x81
    buf = torch.zeros(shift + b.size, dtype=torch.uint8, device="cuda")
    buf[shift:].copy_(torch.from_numpy(b))
    with xe.Correlator(N, C, T, bits=bits, layout=layout) as cor:
        cor.push(buf[shift:])
        vis = cor.dump()
    assert np.array_equal(vis, oracle.correlate(b, N, C, T, bits=bits, layout=layout))


@pytest.mark.parametrize("N,C,T", SHAPES)
@pytest.mark.parametrize("bits,layout", [(4, 0), (4, 1), (4, 2), (8, 0), (8, 1), (8, 2)])
def test_ragged_blocks(N, C, T, bits, layout):
    for shift in (0, 1, 4, 14):
        _push(N, C, T, bits, layout, shift)


@pytest.mark.parametrize("T,pad,skew", [(8, 0, 0), (24, 3, 1), (40, 8, 8), (264, 0, 16), (296, 24, 4), (520, 1, 0)])
def test_packet_turn_strides(T, pad, skew):
    """Every store width, and nothing written past a row's T spectra."""
    import torch
    from paper_1904_07778_gb300.ingest import PacketRing
    F, I, X, K = 3, 5, 2, 9
    pk = synth.random_bytes(T, T * F * I * X * K)
    want = pk.reshape(T // 8, F, X, 8, K, I).transpose(2, 4, 1, 5, 0, 3).reshape(X * K, F * I, T)
    stride = T + pad
    src = torch.zeros(skew + pk.size, dtype=torch.uint8, device="cuda")
    src[skew:].copy_(torch.from_numpy(pk))
    out = torch.full((skew + X * K * F * I * stride + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    with PacketRing(F, I, X, K, T, packet_order=True) as ring:
        ring.turn(src[skew:], out[skew:], out_stride=stride)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    rows = got[skew:skew + X * K * F * I * stride].reshape(X * K, F * I, stride)
    assert np.array_equal(rows[:, :, :T], want)
    assert (rows[:, :, T:] == 0xA5).all() and (got[:skew] == 0xA5).all()
    assert (got[skew + X * K * F * I * stride:] == 0xA5).all()
