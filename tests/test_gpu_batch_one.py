"""One channel per block and one node per thread (batch.cu, the planes at a
constant distance) against packed schedules, bit for bit: a block filled to its
last thread, one node, single rows and columns; odd and even numbers of steps,
within one launch, beyond the replayed graph's 500, and none left over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CHANNELS = [(4, 128, 0.05), (1, 1, 0.3), (512, 1, 1.0), (1, 511, 0.2), (5, 13, 2.5), (31, 16, 0.1)]


@pytest.mark.parametrize("storage", ["fp32s", "fp64"])
@pytest.mark.parametrize("steps", [1, 2, 500, 777])
def test_one_node_per_thread(storage, steps):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    nx, ny, kn = zip(*CHANNELS)
    out = []
    for npt, packed in ((1, 0), (1, 1), (2, 0)):
        b = clb.Batch(list(nx), list(ny), list(kn), g=1e-5, storage=storage, block_x=0)
        b.set_schedule(npt, packed)
        host = np.random.default_rng(5)
        for k in range(len(nx)):
            f = b.state(k)
            b.set_state(k, f * (1 + 0.1 * (2 * host.random(f.shape) - 1)))
        b.step(steps)
        out.append([b.state(k) for k in range(len(nx))])
        b.close()
    for other in out[1:]:
        for x, y in zip(out[0], other):
            assert np.isfinite(x).all()
            np.testing.assert_array_equal(x, y)
