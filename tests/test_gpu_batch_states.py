"""Reading and writing a batch's states, through the transient device buffer of the
first calls and the pinned array of the later ones, and with an allocator that
refuses the transient buffer: the same values, in both storages."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32s", "fp64"])
@pytest.mark.parametrize("n", [2, 30, 70])
def test_states_before_and_after_staging(storage, n):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    ny = [(7 * k) % 40 + 1 for k in range(n)]
    b = clb.Batch([3] * n, ny, [0.2] * n, g=1e-5, storage=storage)
    host = np.random.default_rng(n)
    want = [host.uniform(0.9, 1.1, (9, ny[k], 3)) / 9 for k in range(n)]
    for _ in range(2):
        for k in range(n):
            b.set_state(k, want[k])
        got = [b.state(k) for k in range(n)]
        for x, y in zip(got, want):
            np.testing.assert_allclose(x, y, rtol=0 if storage == "fp64" else 2e-7, atol=0 if storage == "fp64" else 2e-8)
    again = [b.state(k % n) for k in range(65)]
    for k, x in enumerate(again):
        np.testing.assert_array_equal(x, got[k % n])
    b.close()
