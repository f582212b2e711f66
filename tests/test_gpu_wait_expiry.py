"""A grid barrier whose bounded wait runs out (the test hook lp_hold_barrier makes it wait
for arrivals that never come): every call that launches such a kernel returns
LP_ERR_TIMEOUT, leaves nothing half-done behind, and the handle works again afterwards."""
import numpy as np
import pytest

from paper_2105_12715_gb300 import lpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lpm():
    import torch

    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2105_12715_gb300 import lp

    lp.load()
    return lp


M, N = 5000, 25000
DATA = lpgen.large_mixed(4, m=M, n=N)


def hold(lpm, g, on):
    assert lpm.load().lp_hold_barrier(g.h, on) == lpm.LP_OK


def expect(lpm, status, call, *args):
    with pytest.raises(lpm.LPError) as e:
        call(*args)
    assert e.value.status == status


def make(lpm, k):
    return lpm.LP(DATA, eta=0.05, check_every=k, max_iter=6 * k, omega=0.5)


def same(a, b):
    for k in b:
        np.testing.assert_array_equal(a[k], b[k], err_msg=str(k))


def gradient(lpm, g):
    rng = np.random.default_rng(2)
    dc, db = np.empty(N), np.empty(M)
    lpm.lp_backward(g.h, rng.standard_normal(N), rng.standard_normal(M), dc, db)
    return {"dc": dc, "db": db}


# K = 16: the resident kernel on the grid; K = 1025: per-pass kernels, the search's barrier
@pytest.mark.parametrize("k", [16, 1025])
def test_solve(lpm, k):
    with make(lpm, k) as g:
        assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
        fresh = g.state()
        g.set_state()
        hold(lpm, g, 1)
        expect(lpm, lpm.LP_ERR_TIMEOUT, g.solve, 1e-300)
        assert g.info().status == lpm.LP_ERR_TIMEOUT
        hold(lpm, g, 0)
        g.set_state()
        assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
        same(g.state(), fresh)


@pytest.mark.parametrize("k", [16, 1025])
@pytest.mark.parametrize("blocks", [1, 3])
def test_recorded_solve(lpm, k, blocks):
    """The first block expires, which for blocks = 1 is also the last."""
    with make(lpm, k) as g:
        lpm.lp_solve_recorded(g.h, blocks * k)
        fresh = gradient(lpm, g)
        g.set_state()
        hold(lpm, g, 1)
        expect(lpm, lpm.LP_ERR_TIMEOUT, lpm.lp_solve_recorded, g.h, blocks * k)
        expect(lpm, lpm.LP_ERR_NOT_SOLVED, gradient, lpm, g)  # no recording is kept
        hold(lpm, g, 0)
        g.set_state()
        lpm.lp_solve_recorded(g.h, blocks * k)
        same(gradient(lpm, g), fresh)


def test_backward(lpm):
    with make(lpm, 16) as g:
        lpm.lp_solve_recorded(g.h, 64)
        fresh = gradient(lpm, g)
        hold(lpm, g, 1)
        expect(lpm, lpm.LP_ERR_TIMEOUT, gradient, lpm, g)
        hold(lpm, g, 0)
        same(gradient(lpm, g), fresh)


def test_select_omega(lpm):
    """No candidate is ranked by a check that did not happen; the handle keeps its weight,
    its restart scheme and its starting point."""
    grid = [0.25, 1.0, 4.0]
    with make(lpm, 16) as g:
        best, kkt = g.select_omega(grid, iters=96)
    with make(lpm, 16) as g:
        assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
        fresh, restarts = g.state(), g.info().restarts
        assert restarts > 0
        hold(lpm, g, 1)
        expect(lpm, lpm.LP_ERR_TIMEOUT, g.select_omega, grid, 96)
        hold(lpm, g, 0)
        assert g.info().omega == 0.5 and g.info().iters == 0
        assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
        assert g.info().restarts == restarts
        same(g.state(), fresh)
        again = g.select_omega(grid, iters=96)
        assert again[0] == best
        np.testing.assert_array_equal(again[1], kkt)
