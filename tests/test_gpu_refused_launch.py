"""A device that refuses the resident kernel's launch (the test hooks ask for more shared
memory than a block may have, which the host turns into an error at capture): the handle
takes the per-pass kernels, with the same iterates and gradients."""
import numpy as np
import pytest

from paper_2105_12715_gb300 import lpgen

pytestmark = pytest.mark.gpu

OPTS = dict(eta=0.05, check_every=16, max_iter=16 * 7)


@pytest.fixture(scope="module")
def lpm():
    import torch

    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2105_12715_gb300 import lp

    lp.load()
    return lp


# one cluster; the grid (a cooperative launch)
@pytest.mark.parametrize("m,n", [(200, 400), (2000, 9000)])
@pytest.mark.parametrize("precision", [0, 1])
def test_single(lpm, m, n, precision):
    data = lpgen.large_mixed(3, m=m, n=n)
    out = []
    for refuse in (0, 1):
        with lpm.LP(data, autotune=1, precision=precision, **OPTS) as g:
            if refuse:
                assert lpm.load().lp_refuse_resident(g.h) == lpm.LP_OK
            assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
            assert (g.info().graph_kernels > 1) == bool(refuse)
            out.append(g.state())
    for k in out[0]:
        np.testing.assert_array_equal(out[1][k], out[0][k], err_msg=k)


@pytest.mark.parametrize("precision", [0, 1])
def test_batch(lpm, precision):
    probs = [lpgen.large_mixed(k, m=100 + k, n=300) for k in range(30)]
    out = []
    for refuse in (0, 1):
        with lpm.LPBatch(probs, autotune=1, precision=precision, **OPTS) as g:
            if refuse:
                assert lpm.load().lp_batch_refuse_resident(g.h) == lpm.LP_OK
            assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
            out.append((g.state(), [(p["iters"], p["restarts"]) for p in g.info()[1]]))
    for k in out[0][0]:
        np.testing.assert_array_equal(out[1][0][k], out[0][0][k], err_msg=k)
    assert out[1][1] == out[0][1]


def test_batch_backward(lpm):
    probs = [lpgen.large_mixed(k, m=100 + k, n=300) for k in range(30)]
    rng = np.random.default_rng(3)
    wx, wy = rng.standard_normal(30 * 300), rng.standard_normal(sum(p.m for p in probs))
    out = []
    for refuse in (0, 1):
        with lpm.LPBatch(probs, autotune=1, **OPTS) as g:
            if refuse:
                assert lpm.load().lp_batch_refuse_resident(g.h) == lpm.LP_OK
            g.solve_recorded(64)
            out.append(g.backward(wx, wy))
    # the two backward paths contract the recurrence's products into FMAs differently
    for a, b in zip(*out):
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-12 * max(1.0, np.abs(b).max()))
