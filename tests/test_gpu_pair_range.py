"""FP64 channels given numbers that the collision in FP32 pairs cannot take: they
must collide in plain FP64, as the oracle does, on every engine.

The centreline density of a column (kn_mode 1) of one that has diverged: rows out
of the streaming's reach of the bad node become non-finite with it at once, or,
where it is finite, follow it as the oracle does (1e-12, the tolerance of FP64
parity)."""
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


@pytest.mark.parametrize("pipeline", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e40, -3.0])
def test_centre_density_out_of_range(clb, oracle_mod, pipeline, bad):
    nx, ny, xb, yc = 40, 9, 17, 4
    ch = clb.Channel(nx, ny, 0.2, drive="pressure", drive_value=1.5, storage="fp64", kn_mode=1, pipeline=pipeline)
    orc = oracle_mod.OracleSim(oracle_mod.OracleParams(nx=nx, ny=ny, pressure=True, kn=0.2, rho_in=1.5, kn_mode=1))
    f = inputs.perturb(inputs.rng(3), orc.state(), 0.01)
    f[:, yc, xb] = bad / 9
    ch.set_state(f)
    orc.set_state(f)
    ch.step(1)
    orc.step(1)
    got, want = ch.state(), orc.state()
    far = [0, 1, 2, 6, 7, 8]
    if np.isfinite(bad):
        assert np.isfinite(want[:, far]).all()
        assert (np.abs(got[:, far] - want[:, far]) / np.abs(want[:, far])).max() <= 1e-12
    else:  # (the oracle's quotients turn an infinite density into finite rates)
        assert not np.isfinite(got[:, far, xb]).any()
        rest = np.arange(nx) != xb
        assert (np.abs(got - want)[:, far][:, :, rest] / np.abs(want[:, far][:, :, rest])).max() <= 1e-12
    ch.close()


@pytest.mark.parametrize("pipeline", [0, 1])
@pytest.mark.parametrize("kn", [1e-45, 1e-39, 1e-14, 1e12, 1e38, 1e100])
def test_rate_constants_out_of_range(clb, oracle_mod, pipeline, kn):
    """Knudsen numbers whose constants no FP32 number holds, and those beside them."""
    nx, ny = 40, 9
    ch = clb.Channel(nx, ny, kn, drive="pressure", drive_value=1.5, storage="fp64", pipeline=pipeline)
    orc = oracle_mod.OracleSim(oracle_mod.OracleParams(nx=nx, ny=ny, pressure=True, kn=kn, rho_in=1.5))
    f = inputs.perturb(inputs.rng(4), orc.state(), 0.01)
    ch.set_state(f)
    orc.set_state(f)
    ch.step(2)
    orc.step(2)
    want = orc.state()
    assert (np.abs(ch.state() - want) / np.abs(want)).max() <= 1e-12
    ch.close()


def test_force_out_of_range(clb, oracle_mod):
    """A body force beyond FP32: the step that has it is the plain one, without an infinity."""
    ch = clb.Channel(6, 9, 0.2, drive="body_force", drive_value=1e60, storage="fp64")
    orc = oracle_mod.OracleSim(oracle_mod.OracleParams(nx=6, ny=9, kn=0.2, gx=1e60))
    f = inputs.perturb(inputs.rng(5), orc.state(), 0.01)
    ch.set_state(f)
    orc.set_state(f)
    ch.step(1)
    orc.step(1)
    got, want = ch.state(), orc.state()
    assert np.isfinite(want).all()
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    ch.close()
