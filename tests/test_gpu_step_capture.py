"""clb_step captured by the caller (calls that replay no chunk of their own): a
captured call of an even number of steps ends on the buffer it started from,
whatever number of launches takes it, so that replaying it advances the channel
by that many steps each time, bit for bit as calls do."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,drive,storage,kn_mode,kw", [
    (801, 8, "pressure", "fp32s", 0, {}), (801, 8, "pressure", "fp64", 1, {}), (1601, 16, "body_force", "fp16s", 0, {}),
    (4, 32, "body_force", "fp32s", 0, {}), (4, 32, "body_force", "fp64", 0, {}), (16, 16, "body_force", "bf16s", 0, {}),
    (8001, 64, "pressure", "fp32s", 0, {}), (6401, 64, "pressure", "fp32s", 0, {}), (801, 8, "pressure", "fp32s", 0, dict(pipeline=1))])
@pytest.mark.parametrize("n", [2, 4, 10, 30])
def test_replayed_capture_advances(nx, ny, drive, storage, kn_mode, kw, n):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    def make():
        return clb.Channel(nx, ny, 0.2, drive=drive, drive_value=1.8 if drive == "pressure" else 1e-5, storage=storage,
                           kn_mode=kn_mode, **kw)

    ref, ch = make(), make()
    ref.step(3 * n)
    want = ref.state()
    start = ch.state()
    ch.step(n)  # (the kernels are loaded)
    ch.set_state(start)
    ch.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=ch.stream, capture_error_mode="relaxed"):
        ch.step(n)
    with torch.cuda.stream(ch.stream):
        for _ in range(3):
            graph.replay()
    np.testing.assert_array_equal(ch.state(), want)
    ch.close()
    ref.close()
