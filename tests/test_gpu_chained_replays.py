"""Long runs of launches that each start while the previous one drains, on the
plans where many blocks of consecutive launches share the SMs and read halo
columns that other SMs have just written (tile.cu, small planes), and on the
two-step and TMA-staged sweeps: the same bits as the direct sweep after
thousands of steps, replayed and launched one by one."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,drive,storage,steps", [
    (1601, 16, "pressure", "fp32s", 6000), (801, 8, "pressure", "fp32s", 6000), (801, 8, "pressure", "fp64", 2000),
    (2101, 17, "body_force", "fp32s", 4000), (1201, 12, "body_force", "fp16s", 4000), (8001, 64, "pressure", "fp32s", 501),
    (10001, 107, "pressure", "fp16s", 301)])
def test_long_chains_bitwise_equal_direct(nx, ny, drive, storage, steps):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    chans = [clb.Channel(nx, ny, 0.2, drive=drive, drive_value=1.8 if drive == "pressure" else 1e-5, storage=storage,
                         **kw) for kw in (dict(pipeline=1), dict(), dict(graph_steps=-1))]
    f0 = inputs.perturb(inputs.rng(nx + ny), chans[0].state(), 0.02)
    for c in chans:
        c.set_state(f0)
        c.step(steps)
    want = chans[0].state()
    assert np.isfinite(want).all()
    for c in chans[1:]:
        np.testing.assert_array_equal(c.state(), want)
    for c in chans:
        c.close()
