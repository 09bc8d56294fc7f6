"""Objects of different sizes held together: the shared memory a kernel may take
is set per kernel and process, so creating or running one object must not take
it from another, in either order of creation, launched one by one or replayed,
or from another thread.  Every object gives the bits it gives alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clb():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    return clb


SIZES = {"pressure": [(801, 8), (1601, 16), (2101, 21), (2401, 24), (401, 8)],
         "body_force": [(801, 8), (1601, 16), (701, 5), (4, 32), (40, 31)]}


@pytest.mark.parametrize("storage", ["fp32s", "fp16s", "bf16s", "fp64"])
@pytest.mark.parametrize("drive", ["pressure", "body_force"])
def test_tiled_channels_together(clb, storage, drive):
    def make(nx, ny, **kw):
        return clb.Channel(nx, ny, 0.2, drive=drive, drive_value=1.8 if drive == "pressure" else 1e-5, storage=storage, **kw)

    want = {}
    for size in SIZES[drive]:
        ch = make(*size, pipeline=1)
        ch.step(213)
        want[size] = ch.state()
        ch.close()
    for order in (SIZES[drive], SIZES[drive][::-1]):
        chans = {size: make(*size) for size in order}
        for n in (3, 200, 10):
            for ch in chans.values():
                ch.step(n)
        for size, ch in chans.items():
            np.testing.assert_array_equal(ch.state(), want[size])
            ch.close()


@pytest.mark.parametrize("storage", ["fp32s", "fp64"])
def test_batches_together(clb, storage):
    shapes = [dict(nx=[4] * 3, ny=[300, 128, 40], kn=[0.1, 0.3, 1.0]), dict(nx=[4, 3], ny=[32, 16], kn=[0.2, 0.5]),
              dict(nx=[4] * 2, ny=[200, 64], kn=[0.05, 2.0])]

    def make(schedule, **kw):
        b = clb.Batch(kw["nx"], kw["ny"], kw["kn"], g=1e-5, storage=storage)
        if schedule:
            b.set_schedule(*schedule)
        else:
            b.tune()
        return b

    def states(b):
        out = [b.state(k) for k in range(b.n)]
        b.close()
        return out

    want = []
    for kw in shapes:
        b = make((8, 0), **kw)
        b.step(613)
        want.append(states(b))
    for schedule in ((8, 0), (4, 1), None):
        for order in ((0, 1, 2), (2, 1, 0)):
            batches = {k: make(schedule, **shapes[k]) for k in order}
            for n in (3, 600, 10):
                for b in batches.values():
                    b.step(n)
            for k, b in batches.items():
                for x, y in zip(states(b), want[k]):
                    np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("storage,grids", [("fp32s", [(4, 64), (2, 9), (100, 50), (20, 40)]),
                                           ("fp64", [(31, 45), (4, 64), (2, 9), (12, 30)])])
def test_gradients_in_threads(clb, storage, grids):
    def gradient(nx, ny):
        fg = clb.FlowGradient(nx, ny, 0.3, 2.0, 0.8, 2e-5, 40, storage=storage)
        out = (fg.J, *fg.grad())
        fg.close()
        return out

    want = {g: gradient(*g) for g in grids}
    wrong = []

    def work(g):
        try:
            for _ in range(60):
                got = gradient(*g)
                if got != want[g]:
                    wrong.append((g, got))
        except Exception as e:  # noqa: BLE001 - reported below, in the test's own thread
            wrong.append((g, repr(e)))

    threads = [threading.Thread(target=work, args=(g,)) for g in grids]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:4]
