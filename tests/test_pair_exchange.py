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
