"""Calls of one step, two and a few on channels that take several steps per launch:
short calls are left to the direct sweep, and any sequence of calls gives its
bits, with the centreline density carried from one engine to the other."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32s", "fp16s", "fp64"])
@pytest.mark.parametrize("nx,ny,drive,kn_mode", [
    (4, 32, "body_force", 0), (16, 16, "body_force", 0), (1, 16, "body_force", 0), (801, 8, "pressure", 1),
    (401, 17, "pressure", 1), (2101, 33, "body_force", 0), (12, 5, "pressure", 1)])
def test_short_calls(storage, nx, ny, drive, kn_mode):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    a, b = (clb.Channel(nx, ny, 0.2, drive=drive, drive_value=1.3 if drive == "pressure" else 1e-5, storage=storage,
                        kn_mode=kn_mode, **kw) for kw in (dict(), dict(pipeline=1)))
    f0 = inputs.perturb(inputs.rng(nx + ny), b.state(), 0.02)
    for c in (a, b):
        c.set_state(f0)
        for n in (1, 1, 2, 5, 1, 3, 2, 2, 4, 1, 70, 1, 2, 7):
            c.step(n)
    assert a.info()["step"] == 102
    np.testing.assert_array_equal(a.state(), b.state())
    for c in (a, b):
        c.close()
