"""Failure detection of the bounded device-side waits at 8 bits, with one CTA
a task and with pairs of CTAs: a load that nothing will ever deliver makes the
waits of the CTA, and in a pair those of the other CTA that depend on it, run
out within the limit asked for; every role of both CTAs leaves, the dump
reports the timeout, and the same context then integrates a block exactly."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1904_07778_gb300 import synth  # noqa: E402


# stages of 64 spectra (128 where A = B); the withheld stage is the first, one
# within the ring's depth, one whose accumulator is the first buffer's second
# use, and a later task's
@pytest.mark.parametrize("N,C,T,stage", [(192, 4, 1024, 2), (64, 8, 2048, 0), (256, 2, 1024, 0), (256, 3, 1024, 5),
                                         (512, 2, 4096, 40), (320, 200, 64, 2)])
@pytest.mark.parametrize("layout", [0, 2])
def test_withheld_stage_at_8_bits(N, C, T, stage, layout):
    from paper_1904_07778_gb300 import xengine as xe
    blocks = []
    for k in range(2):
        b = synth.random_bytes(70 + k, 2 * N * C * T)
        b[b == 0x80] = 0x81
        blocks.append(b)
    dev = [torch.from_numpy(b).cuda() for b in blocks]
    with xe.Correlator(N, C, T, bits=8, layout=layout) as cor:
        cor.push(dev[0])
        cor.dump()
        cor.set_fault_injection(stage, wait_log2=22)            # about 2 ms per wait
        t0 = time.perf_counter()
        cor.push(dev[0])
        cor.dump(check=False)
        elapsed = time.perf_counter() - t0
        assert cor.last_status == xe.CORR_ETIMEDOUT
        assert elapsed < 0.5                                    # the full limit is a second a wait
        cor.set_fault_injection(-1, 0)
        cor.push(dev[1])
        vis = cor.dump()                                        # raises on a non-OK status
    c = C - 1
    x = blocks[1].reshape((T, C, N, 2) if layout == 0 else (C, N, T, 2))
    one = np.ascontiguousarray(x[:, c] if layout == 0 else x[c])
    assert np.array_equal(vis[c:], oracle.correlate(one, N, 1, T, bits=8, layout=layout))


@pytest.mark.parametrize("N,C,T,bits", [(32, 64, 1024, 4), (192, 8, 2048, 4), (192, 4, 1024, 8), (256, 8, 1024, 8)])
@pytest.mark.parametrize("wait_log2", [1, 9, 12])
def test_limits_shorter_than_a_load(N, C, T, bits, wait_log2):
    """Limits that run out while loads and MMAs are in flight: the roles give
    up, what is in flight still lands before the CTA leaves, and the next
    integration is exact."""
    from paper_1904_07778_gb300 import xengine as xe
    b = synth.random_bytes(5 + N, N * C * T * bits // 4)
    b[b == 0x80] = 0x81
    dev = torch.from_numpy(b).cuda()
    want = oracle.correlate(b, N, C, T, bits=bits, layout=2)
    with xe.Correlator(N, C, T, bits=bits, layout=2) as cor:
        for _ in range(20):
            cor.set_fault_injection(-1, wait_log2=wait_log2)
            cor.push(dev)
            vis = cor.dump(check=False)
            assert cor.last_status in (xe.CORR_OK, xe.CORR_ETIMEDOUT)
            assert cor.last_status == xe.CORR_ETIMEDOUT or np.array_equal(vis, want)
            cor.set_fault_injection(-1, 0)
            cor.push(dev)
            assert np.array_equal(cor.dump(), want)
