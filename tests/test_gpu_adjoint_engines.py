"""The adjoint's engines on grids at the edges of their ranges (one column, one
row, the last grid of one node per thread and the first beyond it, the first
whose forward pass takes a cluster, the last of the cluster and the first with
one launch per step) against one launch per step.  Every engine computes the
same states; the adjoint of a node is the same expression in each, which the
compiler may contract differently, and the sums are taken in another order:
1e-12 in FP64, 1e-5 in FP32, as for the resident engine of small grids."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clb():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    return clb


@pytest.mark.parametrize("storage,tol,nx,ny,n,every", [
    ("fp32s", 1e-5, 1, 1, 60, 7), ("fp32s", 1e-5, 9, 1, 60, 0), ("fp32s", 1e-5, 1, 33, 300, 300),
    ("fp32s", 1e-5, 16, 32, 200, 17), ("fp32s", 1e-5, 19, 27, 200, 17), ("fp32s", 1e-5, 25, 41, 200, 400),
    ("fp32s", 1e-5, 91, 90, 120, 11), ("fp32s", 1e-5, 128, 192, 60, 0), ("fp32s", 1e-5, 173, 143, 60, 0),
    ("fp64", 1e-12, 1, 1, 60, 7), ("fp64", 1e-12, 4, 32, 200, 17), ("fp64", 1e-12, 3, 43, 200, 17),
    ("fp64", 1e-12, 31, 45, 60, 0), ("fp64", 1e-12, 40, 40, 40, 0),
    # a cluster with a node per thread: full blocks, one node more per block than
    # that, shares by columns, blocks left without nodes, single rows and columns
    ("fp32s", 1e-5, 96, 64, 60, 0), ("fp32s", 1e-5, 97, 64, 60, 0), ("fp32s", 1e-5, 100, 50, 90, 13),
    ("fp32s", 1e-5, 40, 33, 90, 1), ("fp32s", 1e-5, 6000, 1, 60, 0), ("fp32s", 1e-5, 1, 600, 90, 7),
    ("fp32s", 1e-5, 3000, 2, 60, 0), ("fp64", 1e-12, 100, 12, 40, 7), ("fp64", 1e-12, 300, 1, 40, 40)])
def test_engines_match_one_launch_per_step(clb, storage, tol, nx, ny, n, every):
    out = []
    for pipeline in (0, 1):
        fg = clb.FlowGradient(nx, ny, 0.3, 2.0, 0.8, 2e-5, n, storage=storage, checkpoint_every=every,
                              pipeline=pipeline)
        out.append((fg.J, *fg.grad()))
        fg.close()
    assert out[0] == pytest.approx(out[1], rel=tol)


def test_second_segment_refused(clb):
    """The pair of blocks holds two segments, or one where the allocator
    refuses the second: the same gradient, bit for bit."""
    import torch

    def run(limit):
        refused = []

        def alloc(n, ctx):
            if n > limit:
                refused.append(n)
                return None
            return torch.cuda.caching_allocator_alloc(int(n))

        def free(p, ctx):
            torch.cuda.caching_allocator_delete(int(p))

        o = clb.clb_opts_default()
        hooks = (clb.ALLOC_FN(alloc), clb.FREE_FN(free))
        o.alloc, o.free = hooks
        h, J = clb.clb_adjoint_forward(4, 16, 0.3, 2.0, 0.8, 2e-5, 500, 50, o)
        g = clb.clb_adjoint_backward(h)
        clb.clb_adjoint_destroy(h)
        return J, g, len(refused)

    one_segment = 4 * 50 * (9 * 64 + 8 * 4)
    J, g, refused = run(1 << 40)
    assert refused == 0
    J1, g1, refused = run(2 * one_segment - 1)
    assert refused == 1
    assert (J1, g1) == (J, g)


def test_wall_terms_refused(clb):
    """A segment of pulled populations and wall terms is larger than its plain
    states where the grid is wide: the cluster, which keeps the states, takes
    the backward pass where the allocator refuses the former."""
    import torch

    def run(limit):
        refused = []

        def alloc(n, ctx):
            if n > limit:
                refused.append(n)
                return None
            return torch.cuda.caching_allocator_alloc(int(n))

        def free(p, ctx):
            torch.cuda.caching_allocator_delete(int(p))

        o = clb.clb_opts_default()
        hooks = (clb.ALLOC_FN(alloc), clb.FREE_FN(free))
        o.alloc, o.free = hooks
        h, J = clb.clb_adjoint_forward(16, 4, 0.3, 2.0, 0.8, 2e-5, 500, 50, o)
        g = clb.clb_adjoint_backward(h)
        clb.clb_adjoint_destroy(h)
        return (J, *g), len(refused)

    want, refused = run(1 << 40)
    assert refused == 0
    got, refused = run(4 * 51 * 9 * 64)
    assert refused == 2
    assert got == pytest.approx(want, rel=1e-5)
