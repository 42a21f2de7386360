"""The padded rows of a 4-bit [c][i][t] context, an extra buffer that only
makes pushes faster, never cost it a call: an allocation that fails beside
them takes their memory, and pushes go on without them, with the same sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1904_07778_gb300 import synth  # noqa: E402

N, C, T = 64, 512, 1001     # 32.8 MB a block, 33.6 MB padded, 17 MB of visibilities


def _fill():
    """Device memory taken in ever smaller pieces until not even 10 MB fit."""
    held, size = [], 1 << 38
    while size >= 10 << 20:
        try:
            held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.cuda.OutOfMemoryError:
            size //= 2
    return held


@pytest.mark.parametrize("what", ["stage", "async"])
def test_padded_rows_give_way(what):
    from paper_1904_07778_gb300 import xengine as xe
    blk = synth.random_bytes(11, N * C * T)
    want = oracle.correlate(blk, N, C, T, layout=xe.CORR_L_CIT)
    dev = torch.from_numpy(blk).cuda()
    # every kernel of this test loaded before memory is short: a block at an odd
    # address goes through plain loads
    odd = torch.zeros(N * C * 16 + 1, dtype=torch.uint8, device="cuda")
    with xe.Correlator(N, C, 16, bits=4, layout=xe.CORR_L_CIT) as w:
        w.push(odd[1:])
        w.push(synth.random_bytes(1, N * C * 16))
        w.dump()
    out = torch.zeros((C, N * (N + 1) // 2, 2), dtype=torch.int64, device="cuda")
    with xe.Correlator(N, C, T, bits=4, layout=xe.CORR_L_CIT) as cor:
        cor.push(dev)
        assert np.array_equal(cor.dump(), want)
        assert cor.stats()["turn_launches"] == 1            # the padded rows serve
        if what == "async":                                 # its streams, not yet the second accumulator
            cor.dump_async(out, reset=False)
            cor.dump_wait()
            cor.dump()
        held = _fill()
        try:
            if what == "stage":
                cor.push(blk)                               # needs a staging block
                assert cor.stats()["turn_launches"] == 1
                got = cor.dump()
                cor.push(dev)                               # device blocks still go
                assert np.array_equal(cor.dump(), want)
                assert np.array_equal(got, want)
            else:
                cor.push(dev)
                cor.dump_async(out)                         # needs the second accumulator
                cor.dump_wait()
                assert np.array_equal(out.cpu().numpy(), want)
        finally:
            del held
            torch.cuda.empty_cache()


def test_padded_rows_stay_for_a_captured_push():
    """A graph of a push keeps the rows' address: they stay, and replays work."""
    from paper_1904_07778_gb300 import xengine as xe
    blk = synth.random_bytes(12, N * C * T)
    want = oracle.correlate(blk, N, C, T, layout=xe.CORR_L_CIT)
    dev = torch.from_numpy(blk).cuda()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st), xe.Correlator(N, C, T, bits=4, layout=xe.CORR_L_CIT, stream=st.cuda_stream) as cor:
        cor.push(dev)
        cor.dump(reset=False)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            cor.push(dev)                                   # adds the block again
        held = _fill()
        try:
            with pytest.raises(xe.CorrError):
                cor.push(blk)                               # no memory for staging, none given up
        finally:
            del held
            torch.cuda.empty_cache()
        g.replay()
        st.synchronize()
        assert np.array_equal(cor.dump(), 2 * want)
