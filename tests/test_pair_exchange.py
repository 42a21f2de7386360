"""What the two CTAs of a pair (8-bit arrays of more than 192 inputs) exchange
on each other's barriers: arrivals that a CTA waits for, and the last ones,
which have to land before it leaves.  Bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1904_07778_gb300 import synth

pytestmark = pytest.mark.gpu


def _block(seed, n):
    b = synth.random_bytes(seed, n)
    b[b == 0x80] = 0x81
    return b


@pytest.mark.parametrize("N,C,T", [(193, 3, 1), (256, 40, 64), (300, 1, 65), (512, 2, 16)])
def test_pairs_of_one_stage_leave_one_after_the_other(N, C, T):
    """Launches of one or two stages a task, hundreds in a row: a pair's first
    commits are its last ones too, and the next launch's CTAs take its place."""
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    b = _block(N + T, 2 * N * C * T)
    d = torch.from_numpy(b).cuda()
    n = 300
    with xe.Correlator(N, C, T, bits=8, layout=xe.CORR_L_CIT) as cor:
        for _ in range(n):
            cor.push(d)
        vis = cor.dump()
    assert np.array_equal(vis, n * oracle.correlate(b, N, C, T, bits=8, layout=xe.CORR_L_CIT))


@pytest.mark.parametrize("N,C,T,layout", [(512, 4, 4100, 0), (320, 40, 2048, 2)])
def test_long_runs_of_pairs_repeat(N, C, T, layout):
    """Thousands of stages whose operands one CTA of a pair writes and the
    other's MMAs read, accumulators reused every 1024 spectra: every
    integration of one block equals the first, and that the oracle's."""
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    b = _block(N + T, 2 * N * C * T)
    d = torch.from_numpy(b).cuda()
    with xe.Correlator(N, C, T, bits=8, layout=layout) as cor:
        vis = torch.empty((2, C, N * (N + 1) // 2, 2), dtype=torch.int64, device="cuda")
        cor.push(d)
        cor.dump_into(vis[0])
        for _ in range(60):
            cor.push(d)
            cor.dump_into(vis[1])
            assert torch.equal(vis[0], vis[1])
    c = 1 if N == 512 else C // 2   # the oracle: one channel
    x = b.reshape((T, C, N, 2) if layout == 0 else (C, N, T, 2))
    one = np.ascontiguousarray(x[:, c] if layout == 0 else x[c])
    assert np.array_equal(vis[0][c:c + 1].cpu().numpy(), oracle.correlate(one, N, 1, T, bits=8, layout=layout))


@pytest.mark.parametrize("N,C,T", [(257, 149, 256), (257, 150, 256), (257, 150, 257), (385, 200, 128), (385, 200, 129)])
def test_pairs_or_single_ctas_by_size(N, C, T):
    """On both sides of the lines between pairs and single CTAs: one context,
    several blocks a launch, and the service."""
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    b = _block(N + C, 2 * N * C * T)
    d = torch.from_numpy(b).cuda()
    with xe.Correlator(N, C, T, bits=8, layout=xe.CORR_L_CIT) as cor:
        cor.push(d)
        vis = cor.dump()
    x = b.reshape(C, N, T, 2)
    for c in (0, C - 1):
        one = np.ascontiguousarray(x[c])
        assert np.array_equal(vis[c:c + 1], oracle.correlate(one, N, 1, T, bits=8, layout=xe.CORR_L_CIT))
    tci = np.ascontiguousarray(x.transpose(2, 0, 1, 3))
    dt = torch.from_numpy(tci).cuda().view(-1)
    with xe.Correlator(N, C, T, bits=8, layout=xe.CORR_L_TCI) as cor:
        cor.push_many([dt, dt])
        assert np.array_equal(cor.dump(), 2 * vis)
    with xe.Service(1 << 30) as svc:
        rid = svc.submit(N, C, 8, xe.CORR_L_TCI, T, 1)
        torch.cuda.synchronize()
        svc.push(rid, dt)
        svc.tick()
        assert svc.wait() == xe.CORR_OK
        assert np.array_equal(svc.fetch(rid), vis)
