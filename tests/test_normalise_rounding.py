"""corr_normalise where its roundings are decided by exact remainders.

The kernel has the significands of the denominator and of the quotients to
about 2^-45 from float pairs, corrects them by the integer remainder, and where
the correction lies within 2^-10 of half a unit (about 0.2% of all operands)
takes the last step by the sign of the new remainder, which is exact: there is
no operand for which the result may differ from IEEE sqrt and /.  Millions of
seeded operands, thousands of which take that last step in the root and in the
quotients (counted here in integers), are compared bit for bit."""
import math

import numpy as np
import pytest


def _near_half(num, den, bits):
    """Whether num / den (or, without den, sqrt(num)), cut to `bits` significant
    bits, lies within 2^-10 of a unit of half way between two of them."""
    extra = 24
    if den is None:
        k = 2 * (bits + extra) - num.bit_length()
        k += (num.bit_length() + k) & 1
        r = math.isqrt(num << k) if k >= 0 else math.isqrt(num >> -k)
    else:
        k = bits + extra + 1 + den.bit_length() - num.bit_length()
        r = (num << k) // den if k >= 0 else num // (den << -k)
    low = r.bit_length() - bits
    frac = (r & ((1 << low) - 1)) / (1 << low)
    return abs(frac - 0.5) < 2.0 ** -10


def _vis(seed, N, C, power_bits, value_bits):
    rng = np.random.default_rng(seed)
    nbl = N * (N + 1) // 2
    vis = rng.integers(-(1 << value_bits) + 1, 1 << value_bits, (C, nbl, 2))
    d = np.arange(N) * (np.arange(N) + 3) // 2
    vis[:, d, 0] = rng.integers(1, 1 << power_bits, (C, N))
    vis[:, d, 1] = 0
    return vis, d


def _share(vis, d, N, n):
    """Share of near roots and near quotients among the channel 0 baselines' first n."""
    i, j = np.tril_indices(N)
    roots = quots = 0
    for b in range(n):
        den2 = float(vis[0, d[i[b]], 0]) * float(vis[0, d[j[b]], 0])
        m, e = math.frexp(den2)
        m, e = int(m * 2 ** 53), e - 53
        roots += _near_half(m << (e & 1), None, 53)
        s, w = math.sqrt(den2), abs(int(vis[0, b, 0]))
        if w:
            quots += _near_half(w, int(math.frexp(s)[0] * 2 ** 53), 53)
    return roots / n, quots / n


CASES = [(1, 192, 48, 31, 31), (2, 192, 24, 44, 40), (3, 192, 24, 53, 52), (4, 64, 256, 22, 20)]


@pytest.mark.parametrize("seed,N,C,power_bits,value_bits", CASES)
def test_operands_reach_the_last_step(seed, N, C, power_bits, value_bits):
    vis, d = _vis(seed, N, C, power_bits, value_bits)
    roots, quots = _share(vis, d, N, 2000)
    assert 0 < roots < 0.02 and 0 < quots < 0.02


@pytest.mark.gpu
@pytest.mark.parametrize("seed,N,C,power_bits,value_bits", CASES)
def test_last_step_is_ieee(seed, N, C, power_bits, value_bits):
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    vis, d = _vis(seed, N, C, power_bits, value_bits)
    i, j = np.tril_indices(N)
    p = vis[:, d, 0].astype(np.float64)
    want = vis.astype(np.float64) / np.sqrt(p[:, i] * p[:, j])[..., None]
    rho = torch.empty(vis.shape, dtype=torch.float64, device="cuda")
    with xe.Correlator(N, C, 16, bits=4, layout=2) as cor:
        cor.restore(vis)
        cor.normalise_into(rho)
        torch.cuda.synchronize()
    got = rho.cpu().numpy()
    assert np.array_equal(got.view(np.int64), (want + 0.0).view(np.int64))   # + 0.0: the kernel has no -0
