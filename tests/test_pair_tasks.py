"""8-bit arrays of more than 192 inputs, whose tasks are 256 x 256 blocks of
pairs of CTAs: even and odd counts of row blocks and super rows, a row block
of one input, one to several accumulations, every layout, and the calls that
take the tasks another way (several blocks a launch, the pipelined turn, the
service beside small arrays).  Bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1904_07778_gb300 import synth

pytestmark = pytest.mark.gpu


def _block(seed, n):
    b = synth.random_bytes(seed, n)
    b[b == 0x80] = 0x81
    return b


@pytest.mark.parametrize("N,C,T", [(193, 2, 65), (256, 3, 1), (257, 1, 1024), (320, 2, 1025), (321, 1, 128),
                                   (384, 5, 63), (449, 1, 2100), (513, 1, 300)])
@pytest.mark.parametrize("layout", [0, 1, 2])
def test_pair_blocks(N, C, T, layout):
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    b = _block(N + T, 2 * N * C * T)
    with xe.Correlator(N, C, T, bits=8, layout=layout) as cor:
        cor.push(torch.from_numpy(b).cuda())
        cor.push(torch.from_numpy(b).cuda())
        vis = cor.dump()
    assert np.array_equal(vis, 2 * oracle.correlate(b, N, C, T, bits=8, layout=layout))


def test_pair_push_many_and_pipeline():
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    N, C, T = 256, 4, 256
    blocks = [_block(k, 2 * N * C * T) for k in range(3)]
    dev = [torch.from_numpy(b).cuda() for b in blocks]
    want = sum(oracle.correlate(b, N, C, T, bits=8, layout=0) for b in blocks)
    with xe.Correlator(N, C, T, bits=8, layout=0) as cor:
        cor.push_many(dev)
        assert cor.stats()["herk_launches"] == 1
        assert np.array_equal(cor.dump(), want)
        cor.set_pipeline(20)     # single CTAs' tasks beside the turn
        for d in dev:
            cor.push(d)
        assert np.array_equal(cor.dump(), want)
        cor.set_pipeline(0)
        cor.push(dev[0])
        assert np.array_equal(cor.dump(), oracle.correlate(blocks[0], N, C, T, bits=8, layout=0))


def test_pair_requests_beside_small_arrays():
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    shapes = [(320, 3, 512), (192, 4, 512), (32, 8, 512), (200, 2, 1200)]
    with xe.Service(1 << 30) as svc:
        ids = [svc.submit(n, c, 8, 0, t, 2) for n, c, t in shapes]
        want = [None] * len(shapes)
        for k in range(2):
            for q, (n, c, t) in enumerate(shapes):
                b = _block(10 * k + q, 2 * n * c * t)
                d = torch.from_numpy(b).cuda()
                torch.cuda.synchronize()
                svc.push(ids[q], d)
                svc.wait()
                v = oracle.correlate(b, n, c, t, bits=8, layout=0)
                want[q] = v if want[q] is None else want[q] + v
            assert svc.tick() == len(shapes)
        assert svc.wait() == xe.CORR_OK
        for q in range(len(shapes)):
            assert np.array_equal(svc.fetch(ids[q]), want[q])
