"""How a channelise call is cut into groups of spectra changes nothing: one
call over T spectra (32, 16, 8 ... spectra per FFT unit, as the size allows)
equals the same spectra in short calls (two per unit), bit for bit, for gains
on both sides of the bound where the equaliser needs no clamp."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,T,taps,low_gain", [
    (192, 1024, 451, 4, False), (192, 64, 3700, 4, True), (192, 128, 1001, 3, False),
    (100, 512, 200, 4, True), (191, 256, 300, 4, False), (192, 64, 3605, 6, False)])
@pytest.mark.parametrize("layout", [0, 2])
def test_one_call_is_its_slices(N, C, T, taps, low_gain, layout):
    import torch
    from paper_1904_07778_gb300.fengine import FEngine
    M = 2 * C
    g = torch.Generator(device="cuda").manual_seed(N + T)
    adc = torch.randint(-127, 128, (N, (T + taps - 1) * M), generator=g, device="cuda", dtype=torch.int8)
    gain = np.random.default_rng(T).integers(120, 6000, (C, N)).astype(np.uint32)
    if low_gain:
        gain[::3] = np.random.default_rng(C).integers(0, 140, gain[::3].shape)
    gain[1, 0] = 0
    with FEngine(N, C, taps) as f:
        f.set_gains(gain)

        def call(t0, n, stride):
            out = torch.zeros((C, N, stride) if layout == 2 else (n, C, N), dtype=torch.uint8, device="cuda")
            power = torch.zeros((C, N), dtype=torch.int64, device="cuda")
            part = adc[:, t0 * M:(t0 + n + taps - 1) * M].contiguous()
            f.channelise(part, n, out=out, layout=layout, out_stride=stride)
            f.channelise(part, n, out=None, power=power)
            f.sync()
            return out, power

        stride = (T + 15) // 16 * 16
        whole, power = call(0, T, stride)
        total = torch.zeros_like(power)
        step = 24
        for t0 in range(0, T, step):
            n = min(step, T - t0)
            part, p = call(t0, n, 24)
            total += p
            if layout == 2:
                assert torch.equal(whole[:, :, t0:t0 + n], part[:, :, :n]), t0
            else:
                assert torch.equal(whole[t0:t0 + n], part), t0
        assert torch.equal(power, total)
        if layout == 2:
            assert int(whole[:, :, T:].count_nonzero()) == 0   # nothing past the spectra


@pytest.mark.parametrize("N,C,T,taps", [(3, 1024, 37, 4), (2, 2048, 5, 4), (5, 64, 333, 4), (1, 256, 131, 3),
                                        (3, 512, 70, 16), (2, 16, 1000, 1)])
@pytest.mark.parametrize("low_gain", [False, True])
def test_powers_of_saturating_spectra(N, C, T, taps, low_gain):
    """Full-scale constant and alternating inputs, past the 18-bit range where
    the transform is long enough: the power sums are those of the 18-bit
    values, over every unit of a CTA, and add to what is there; the codes do
    not depend on whether powers are asked for."""
    import torch
    from paper_1904_07778_gb300.fengine import FEngine
    M = 2 * C
    rng = np.random.default_rng(C + T)
    S = (T + taps - 1) * M
    adc = rng.integers(-20, 21, (N, S)).astype(np.int8)
    adc[0] = 127
    if N > 1:
        adc[1] = np.where(np.arange(S) % 2, -127, 127)
    gain = rng.integers(0, 140, (C, N)) if low_gain else rng.integers(120, 6000, (C, N))
    adc = torch.from_numpy(adc).cuda()
    with FEngine(N, C, taps) as f:
        f.set_gains(gain.astype(np.uint32))
        v18 = torch.empty((T, C, N, 2), dtype=torch.int32, device="cuda")
        plain = torch.zeros((T, C, N), dtype=torch.uint8, device="cuda")
        f.channelise(adc, T, out=plain, layout=0, v18=v18)
        power = torch.full((C, N), 5, dtype=torch.int64, device="cuda")
        codes = torch.zeros_like(plain)
        f.channelise(adc, T, out=codes, layout=0, power=power)
        f.sync()
    v = v18.long()
    if C >= 1024:
        assert int(v.max()) == 131071
    assert torch.equal(power, (v * v).sum(dim=(0, 3)) + 5)
    assert torch.equal(codes, plain)


@pytest.mark.parametrize("N,C,T", [(3, 64, 2), (2, 64, 7), (5, 128, 67), (4, 64, 1030), (7, 1024, 45), (2, 2048, 19),
                                   (16, 64, 4099)])
@pytest.mark.parametrize("shift,pad", [(1, 0), (2, 3), (3, 1), (0, 5), (8, 4)])
def test_codes_to_any_address(N, C, T, shift, pad):
    """Rows of codes at any address and stride equal those of aligned rows,
    and nothing is written between them."""
    import torch
    from paper_1904_07778_gb300.fengine import FEngine
    taps, M = 4, 2 * C
    g = torch.Generator(device="cuda").manual_seed(N * C + T)
    adc = torch.randint(-100, 101, (N, (T + taps - 1) * M), generator=g, device="cuda", dtype=torch.int8)
    gain = np.random.default_rng(T).integers(100, 3000, (C, N)).astype(np.uint32)
    stride = (T + 15) // 16 * 16
    with FEngine(N, C, taps) as f:
        f.set_gains(gain)
        want = torch.zeros((C, N, stride), dtype=torch.uint8, device="cuda")
        f.channelise(adc, T, out=want, layout=2, out_stride=stride)
        buf = torch.full((shift + C * N * (T + pad) + 16,), 0x5A, dtype=torch.uint8, device="cuda")
        f.channelise(adc, T, out=buf[shift:], layout=2, out_stride=T + pad)
        f.sync()
    rows = buf[shift:shift + C * N * (T + pad)].view(C, N, T + pad)
    assert torch.equal(rows[:, :, :T], want[:, :, :T])
    assert bool((rows[:, :, T:] == 0x5A).all())
    assert bool((buf[:shift] == 0x5A).all()) and bool((buf[shift + C * N * (T + pad):] == 0x5A).all())


@pytest.mark.parametrize("N,C,T,taps", [(2, 64, 5, 4), (3, 64, 37, 4), (6, 256, 33, 3), (5, 1024, 9, 4), (4, 128, 21, 6)])
@pytest.mark.parametrize("shift", [0, 2])
def test_spectra_and_values_at_any_alignment(N, C, T, taps, shift):
    """The FP32 spectra and 18-bit values, alone and together, at 16- and
    8-byte aligned addresses: the values are the spectra rounded and clamped,
    and the same every way."""
    import torch
    from paper_1904_07778_gb300.fengine import FEngine
    M, n = 2 * C, T * C * N * 2
    g = torch.Generator(device="cuda").manual_seed(N * C + T)
    adc = torch.randint(-127, 128, (N, (T + taps - 1) * M), generator=g, device="cuda", dtype=torch.int8)
    adc[0] = 127
    sp = torch.full((2, n + 8), 7.0, device="cuda")
    v18 = torch.full((2, n + 8), 7, dtype=torch.int32, device="cuda")
    with FEngine(N, C, taps) as f:
        f.set_gains(np.full((C, N), 900, np.uint32))
        f.channelise(adc, T, spec=sp[0, shift:], v18=v18[0, shift:])
        f.channelise(adc, T, spec=sp[1, 4:])
        f.channelise(adc, T, v18=v18[1, 4:])
        f.sync()
    a, v = sp[0, shift:shift + n], v18[0, shift:shift + n]
    assert torch.equal(a, sp[1, 4:4 + n]) and torch.equal(v, v18[1, 4:4 + n])
    assert torch.equal(v, a.double().round().clamp(-131072, 131071).int())
    for buf, s in ((sp[0], shift), (v18[0], shift), (sp[1], 4), (v18[1], 4)):
        assert bool((buf[:s] == 7).all()) and bool((buf[s + n:] == 7).all())
