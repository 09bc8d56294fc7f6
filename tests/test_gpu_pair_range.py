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
