"""Device tensors handed over for a copy on a stream of the library's own: the
copy follows the work queued on the stream that the caller names, and the
tensor's memory is not given to another before the copy is done."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402

SHAPE = (32, 64, 1024, 4, 0)
BYTES = 32 * 64 * 1024


def _samples(seed):
    return np.random.default_rng(seed).integers(0, 256, BYTES, dtype=np.uint8)


@pytest.mark.parametrize("side_stream", [False, True])
def test_batch_input_follows_its_producer(side_stream):
    from paper_1904_07778_gb300 import xengine as xe
    blk = _samples(1)
    src = torch.from_numpy(blk).cuda()
    dst = torch.zeros_like(src)
    with xe.Batch([SHAPE]) as b:
        b.run()
        assert b.sync() == xe.CORR_OK
        torch.cuda.synchronize()
        st = torch.cuda.Stream() if side_stream else torch.cuda.current_stream()
        with torch.cuda.stream(st):
            torch.cuda._sleep(40_000_000)   # the producer is late (about 20 ms)
            dst.copy_(src)
            b.set_input(0, dst, after=torch.cuda.current_stream())
        b.run()
        assert b.sync() == xe.CORR_OK
        assert np.array_equal(b.output(0), oracle.correlate(blk, *SHAPE[:3], layout=0))


def test_batch_input_lives_until_it_is_copied():
    from paper_1904_07778_gb300 import xengine as xe
    blk = _samples(2)
    with xe.Batch([SHAPE, (192, 256, 4096, 4, 0)]) as b:
        b.run()
        assert b.sync() == xe.CORR_OK
        t = torch.from_numpy(blk).cuda()
        torch.cuda.synchronize()
        at = t.data_ptr()
        for _ in range(100):            # the copy waits behind these (some 10 ms)
            b.run()
        b.set_input(0, t)
        del t
        other = [torch.full((BYTES,), 0x77, dtype=torch.uint8, device="cuda") for _ in range(4)]
        assert at not in [o.data_ptr() for o in other]
        b.run()
        assert b.sync() == xe.CORR_OK
        assert np.array_equal(b.output(0), oracle.correlate(blk, *SHAPE[:3], layout=0))


def test_held_inputs_are_let_go():
    """The batch keeps no tensor past the next synchronisation, nor more of
    them than are in flight."""
    import gc
    import weakref
    from paper_1904_07778_gb300 import xengine as xe
    with xe.Batch([SHAPE]) as b:
        refs = []
        for k in range(3):
            x = torch.from_numpy(_samples(5 + k)).cuda()
            refs.append(weakref.ref(x))
            b.set_input(0, x)
            torch.cuda.synchronize()
        del x
        gc.collect()
        assert [r() is None for r in refs] == [True, True, False]   # each call lets earlier ones go
        b.sync()
        gc.collect()
        assert refs[2]() is None
