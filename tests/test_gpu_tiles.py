"""Several steps per launch (tile.cu, the default of small channels) against the
direct sweep (pipeline 1), one launch per step: bit for bit the same
populations, centreline mode and observables, on channels that one block holds
and on channels split into blocks with halos, at the ragged edges of both
(one row, one column, heights around a warp, widths that leave blocks of
unequal size), for every storage and any chunking of the steps; and over a
checkpoint, whose halo columns the next engine reads."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clb():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    return clb


SHAPES = [  # nx, ny, drive, kn_mode
    (1, 7, "body_force", 0), (4, 32, "body_force", 0), (5, 3, "body_force", 0), (4, 2, "pressure", 1),
    (40, 31, "pressure", 0), (700, 1, "body_force", 0), (460, 1, "pressure", 0), (77, 17, "pressure", 1),
    (1601, 16, "pressure", 0), (801, 8, "pressure", 1), (801, 9, "pressure", 1), (2101, 33, "body_force", 0),
    (457, 33, "pressure", 0), (640, 65, "body_force", 0), (3201, 32, "pressure", 0), (2, 300, "body_force", 0),
    (300, 128, "pressure", 0)]


def make(clb, nx, ny, drive, kn_mode, storage, **kw):
    return clb.Channel(nx, ny, 0.2, drive=drive, drive_value=1.8 if drive == "pressure" else 2e-4, storage=storage,
                       kn_mode=kn_mode, **kw)


@pytest.mark.parametrize("storage", ["fp32s", "fp16s", "bf16s", "fp64"])
@pytest.mark.parametrize("nx,ny,drive,kn_mode", SHAPES)
def test_tiles_bitwise_equal_direct(clb, tmp_path, storage, nx, ny, drive, kn_mode):
    ref = make(clb, nx, ny, drive, kn_mode, storage, pipeline=1)
    ch = make(clb, nx, ny, drive, kn_mode, storage)
    f0 = inputs.perturb(inputs.rng(nx * 3 + ny), ref.state(), 0.05)
    ref.set_state(f0)
    ch.set_state(f0)
    for n in (1, 57, 130, 3):
        ref.step(n)
        ch.step(n)
    assert ch.info()["step"] == 191
    np.testing.assert_array_equal(ch.state(), ref.state())
    a, b = ch.observables(check=False), ref.observables(check=False)
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    path = str(tmp_path / "c.clb")
    ch.save(path)
    resumed = clb.Channel.load(path, pipeline=1)
    resumed.step(5)
    ref.step(5)
    np.testing.assert_array_equal(resumed.state(), ref.state())
    for c in (ref, ch, resumed):
        c.close()
