"""corr_normalise against the IEEE evaluation of its definition,
V / sqrt(V_ii V_jj), bit for bit: the kernel's corrected square root and
quotients round as sqrt and / do (each residual is exact, so a result could
only differ if the exact value lay within 2^-48 of an ulp of a rounding
boundary)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _want(vis, N):
    i, j = np.tril_indices(N)
    d = np.arange(N) * (np.arange(N) + 3) // 2
    p = vis[:, d, 0].astype(np.float64)
    with np.errstate(invalid="ignore", divide="ignore"):
        den2 = p[:, i] * p[:, j]
        rho = vis.astype(np.float64) / np.sqrt(den2)[..., None]
    rho[den2 == 0] = 0.0
    return rho, (den2 == 0).astype(np.uint8)


@pytest.mark.parametrize("N,C,mag", [(1, 1, 20), (2, 3, 62), (5, 700, 8), (33, 64, 40), (100, 5, 53),
                                     (257, 2, 30), (1024, 1, 62)])
@pytest.mark.parametrize("skew", [0, 1])
def test_normalise_is_ieee(N, C, mag, skew):
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    rng = np.random.default_rng([N, C, mag])
    nbl = N * (N + 1) // 2
    # magnitudes from 1 to 2^mag, some zero; powers mostly positive, some 0 or negative
    vis = rng.integers(0, 1 << 62, (C, nbl, 2)) >> rng.integers(62 - mag, 63, (C, nbl, 2))
    vis *= rng.choice([-1, 1], vis.shape)
    d = np.arange(N) * (np.arange(N) + 3) // 2
    vis[:, d, 0] = np.abs(vis[:, d, 0]) * rng.choice([1, 1, 1, 1, 0, -1], (C, N))
    want, zf = _want(vis, N)
    # skew: 8-byte aligned output (no 16-byte stores)
    buf = torch.full((C * nbl * 2 + 2,), 7.0, dtype=torch.float64, device="cuda")
    rho = buf[skew:skew + C * nbl * 2]
    flag = torch.full((C * nbl,), 9, dtype=torch.uint8, device="cuda")
    with xe.Correlator(N, C, 16, bits=4, layout=2) as cor:
        cor.restore(vis)
        assert xe.corr_normalise_flags(cor._ctx, rho.data_ptr(), flag.data_ptr()) == xe.CORR_OK
    got = rho.cpu().numpy().reshape(vis.shape)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan], want[~nan])
    assert np.array_equal(flag.cpu().numpy().reshape(C, nbl), zf)
    rest = buf.cpu().numpy()
    assert (np.concatenate([rest[:skew], rest[skew + C * nbl * 2:]]) == 7.0).all()


def test_normalise_at_the_edges():
    """Powers and numerators where the significands change length: powers of
    two and their neighbours, the ends of 32 and 53 bits and of the type."""
    import torch
    from paper_1904_07778_gb300 import xengine as xe
    p = [1, 2, 3, (1 << 24) - 1, (1 << 24) + 1, (1 << 31) - 1, 1 << 31, (1 << 52) - 1, (1 << 53) - 1, (1 << 53) + 1,
         (1 << 62), (1 << 63) - 1, 5, 1 << 40]
    w = [1, 3, (1 << 24) - 1, (1 << 24) + 1, (1 << 31) - 1, 1 << 31, (1 << 31) + 1, (1 << 32) - 1, (1 << 53) - 1, 1 << 53,
         (1 << 53) + 1, (1 << 63) - 1]
    w = np.array([0, -(1 << 63)] + w + [-x for x in w], np.int64)
    N, C = len(p), len(w)
    vis = np.empty((C, N * (N + 1) // 2, 2), np.int64)
    vis[..., 0] = w[:, None]
    vis[..., 1] = np.roll(w, 5)[:, None]
    d = np.arange(N) * (np.arange(N) + 3) // 2
    vis[:, d, 0] = p
    want, _ = _want(vis, N)
    rho = torch.empty(vis.shape, dtype=torch.float64, device="cuda")
    with xe.Correlator(N, C, 16, bits=4, layout=2) as cor:
        cor.restore(vis)
        cor.normalise_into(rho)
        torch.cuda.synchronize()
    assert np.array_equal(rho.cpu().numpy().view(np.int64), want.view(np.int64))
