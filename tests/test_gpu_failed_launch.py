"""A launch that CUDA refuses (here: on a stream whose capture has been
invalidated, which is an error of the call and reaches no GPU) is reported by
that call alone: another channel, created and stepped afterwards, works, and so
does the refused one once the capture has ended."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RELAXED = 2  # CU_STREAM_CAPTURE_MODE_RELAXED


@pytest.mark.parametrize("kw", [dict(pipeline=1), dict(), dict(pipeline=2)], ids=["direct", "tiles", "tma"])
def test_refused_launch_reported_once(kw):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    def make():
        return clb.Channel(801, 12, 0.2, drive="pressure", drive_value=1.8, storage="fp32s", **kw)

    ref = make()
    ref.step(7)
    want = ref.state()
    cu = ctypes.CDLL("libcuda.so.1")
    ch = make()
    ch.sync()
    stream, graph = ctypes.c_void_p(ch.stream.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(stream, RELAXED) == 0
    try:
        assert cu.cuStreamSynchronize(stream) != 0  # not allowed here: invalidates the capture
        with pytest.raises(clb.CLBError) as err:
            ch.step(3)
        assert err.value.status == clb.CLB_ECUDA
    finally:
        assert cu.cuStreamEndCapture(stream, ctypes.byref(graph)) != 0
    other = make()
    for c in (other, ch):
        c.step(7)
        np.testing.assert_array_equal(c.state(), want)
    for c in (ref, ch, other):
        c.close()
