"""Two steps per launch (march.cu, the default of large FP32 pressure channels)
against the direct sweep (pipeline 1): bit for bit the same populations and
observables, with the last column at each place it can have in a lane and in
the halo of the strip before (strips of 120 columns, 4 per lane), with heights
that split into segments of equal and unequal length, one row over a segment,
few rows, and shares that cross from one group of strips to the next; for odd
and even numbers of steps."""
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


@pytest.mark.parametrize("nx,ny", [(2039, 256), (2040, 256), (2041, 257), (2042, 300), (2043, 251), (2044, 250),
                                   (2000, 250), (4097, 128), (16681, 30), (100001, 5), (80001, 13), (500000, 1)])
def test_two_steps_bitwise_equal_direct(clb, nx, ny):
    def make(**kw):
        return clb.Channel(nx, ny, 0.2, drive="pressure", drive_value=1.8, storage="fp32s", **kw)

    ref, ch = make(pipeline=1), make()
    f0 = inputs.perturb(inputs.rng(nx + ny), ref.state(), 0.05)
    ref.set_state(f0)
    ch.set_state(f0)
    for n in (2, 1, 5, 66):
        ref.step(n)
        ch.step(n)
    assert ch.info()["step"] == 74
    np.testing.assert_array_equal(ch.state(), ref.state())
    a, b = ch.observables(check=False), ref.observables(check=False)
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    ref.close()
    ch.close()
