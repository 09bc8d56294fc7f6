"""The adjoint's backward walk over many short segments: the states of a segment
are read by the walk's last terms while other threads are already in the next
segment, so the gradient of a run of one- and two-step segments must have the
same bits every time, and agree with one launch per step (FP32 1e-5, FP64 1e-12,
as for the engines on other grids).  Grids shared over a cluster by columns (wall
terms read a neighbour block's nodes) and by rows."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("every", [1, 2, 3])
@pytest.mark.parametrize("storage,tol,nx,ny", [("fp32s", 1e-5, 100, 50), ("fp32s", 1e-5, 64, 64), ("fp64", 1e-12, 40, 16)])
def test_short_segments_same_bits(storage, tol, nx, ny, every):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    def gradients(repeats, pipeline):
        fg = clb.FlowGradient(nx, ny, 0.3, 2.0, 0.8, 2e-5, 120, storage=storage, checkpoint_every=every, pipeline=pipeline)
        out = [tuple(fg.grad()) for _ in range(repeats)]
        fg.close()
        return out

    got = gradients(60, 0)
    assert set(got) == {got[0]}
    assert got[0] == pytest.approx(gradients(1, 1)[0], rel=tol)
