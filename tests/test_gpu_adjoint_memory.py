"""The adjoint under an allocator with a bounded total: from the first total that
lets a run through to the one that refuses nothing, every total is enough (a
larger segment must not take what a later, smaller buffer needs), and each gives
the same gradient (FP32 1e-5, as for the engines)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 4), (2, 40)])
def test_every_total_above_the_smallest(nx, ny):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1603_01955_gb300.clb as clb

    def run(total):
        used, sizes, refused = [0], {}, []

        def alloc(n, ctx):
            if used[0] + n > total:
                refused.append(n)
                return None
            p = torch.cuda.caching_allocator_alloc(int(n))
            used[0] += n
            sizes[p] = n
            return p

        def free(p, ctx):
            used[0] -= sizes.pop(int(p))
            torch.cuda.caching_allocator_delete(int(p))

        o = clb.clb_opts_default()
        hooks = (clb.ALLOC_FN(alloc), clb.FREE_FN(free))
        o.alloc, o.free = hooks
        h, J = clb.clb_adjoint_forward(nx, ny, 0.3, 2.0, 0.8, 2e-5, 500, 50, o)
        peak = used[0]
        g = clb.clb_adjoint_backward(h)
        clb.clb_adjoint_destroy(h)
        assert used[0] == 0
        return (J, *g), peak, refused

    want, most, refused = run(1 << 40)
    assert not refused
    state = 4 * 9 * nx * ny
    least = (10 + 50 + 4) * state  # ceil(nsteps / C) + C + 4 states, and the partial sums
    wall, pair = 4 * 50 * 8 * nx, 50 * state
    # around every point where a larger segment just fits, in steps of half the partial sums
    for seg in (pair + wall, 2 * (pair + wall)):
        for extra in range(0, 2048, 192):
            total = 13 * state + seg + extra
            if total < least + 1024:
                continue
            got, peak, refused = run(total)
            assert peak <= total
            assert got == pytest.approx(want, rel=1e-5)
