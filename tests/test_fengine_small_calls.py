"""Small channelise calls, on both sides of the rule that gives an FFT unit
two or four spectra: the codes as [c][i][t] rows, in half words, words or
bytes as their alignment allows, are those of the [t][c][i] call, and nothing
is written between the rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,T", [(6, 256, 1024), (6, 256, 1022), (3, 64, 4096), (16, 256, 200), (16, 64, 200),
                                   (64, 64, 128), (64, 64, 127), (2, 2048, 200), (3, 2048, 77), (16, 16, 4096)])
@pytest.mark.parametrize("shift,pad", [(0, 0), (2, 0), (4, 4), (0, 2), (1, 0), (0, 3)])
@pytest.mark.parametrize("extra", [False, True])
def test_rows_are_the_payload_order_codes(N, C, T, shift, pad, extra):
    import torch
    from paper_1904_07778_gb300.fengine import FEngine
    taps, M, stride = 4, 2 * C, T + pad
    g = torch.Generator(device="cuda").manual_seed(N * C + T)
    adc = torch.randint(-90, 91, (N, (T + taps - 1) * M), generator=g, device="cuda", dtype=torch.int8)
    gain = np.random.default_rng(T).integers(100, 3000, (C, N)).astype(np.uint32)
    spec = torch.empty(T * C * N * 2, device="cuda") if extra else None
    with FEngine(N, C, taps) as f:
        f.set_gains(gain)
        want = torch.zeros((T, C, N), dtype=torch.uint8, device="cuda")
        f.channelise(adc, T, out=want, layout=0)
        buf = torch.full((shift + C * N * stride + 16,), 0x5A, dtype=torch.uint8, device="cuda")
        f.channelise(adc, T, out=buf[shift:], layout=2, out_stride=stride, **({"spec": spec} if extra else {}))
        f.sync()
    rows = buf[shift:shift + C * N * stride].view(C, N, stride)
    assert torch.equal(rows[:, :, :T], want.permute(1, 2, 0))
    assert bool((rows[:, :, T:] == 0x5A).all())
    assert bool((buf[:shift] == 0x5A).all()) and bool((buf[shift + C * N * stride:] == 0x5A).all())


@pytest.mark.parametrize("N,C,T", [(191, 64, 10300), (191, 64, 9900), (33, 64, 2048), (191, 256, 128)])
@pytest.mark.parametrize("extra", [False, True])
def test_payload_order_in_either_order_of_ctas(N, C, T, extra):
    """Payload-order outputs below and above the size at which CTAs of
    neighbouring pairs run together: the codes are those of the rows, the
    18-bit values those of a call in parts."""
    import torch
    from paper_1904_07778_gb300.fengine import FEngine
    taps, M = 4, 2 * C
    g = torch.Generator(device="cuda").manual_seed(N * C + T)
    adc = torch.randint(-90, 91, (N, (T + taps - 1) * M), generator=g, device="cuda", dtype=torch.int8)
    gain = np.random.default_rng(T).integers(100, 3000, (C, N)).astype(np.uint32)
    with FEngine(N, C, taps) as f:
        f.set_gains(gain)
        got = torch.zeros((T, C, N), dtype=torch.uint8, device="cuda")
        v18 = torch.empty((T, C, N, 2), dtype=torch.int32, device="cuda") if extra else None
        f.channelise(adc, T, out=got, layout=0, **({"v18": v18} if extra else {}))
        rows = torch.zeros((C, N, T), dtype=torch.uint8, device="cuda")
        f.channelise(adc, T, out=rows, layout=2)
        f.sync()
        assert torch.equal(got, rows.permute(2, 0, 1))
        if extra:
            for t0 in (0, T // 2, T - 5):
                part = torch.empty((5, C, N, 2), dtype=torch.int32, device="cuda")
                f.channelise(adc[:, t0 * M:(t0 + 5 + taps - 1) * M].contiguous(), 5, v18=part)
                f.sync()
                assert torch.equal(part, v18[t0:t0 + 5]), t0
