"""Batches stepped in short and long calls: launches of few steps take another
kernel than long ones, and any sequence of calls gives the bits of one long call
on a schedule that has one kernel only."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32s", "fp64"])
def test_short_and_long_calls(storage):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    nx, ny, kn = [4, 1, 31, 5], [32, 7, 16, 100], [0.1, 1.0, 0.05, 3.0]
    out = []
    for schedule, calls in (((1, 0), (1, 31, 32, 33, 2, 501, 1, 40)), ((2, 1), (641,))):
        b = clb.Batch(nx, ny, kn, g=1e-5, storage=storage)
        b.set_schedule(*schedule)
        for n in calls:
            b.step(n)
        out.append([b.state(k) for k in range(b.n)])
        b.close()
    for x, y in zip(*out):
        assert np.isfinite(x).all()
        np.testing.assert_array_equal(x, y)
