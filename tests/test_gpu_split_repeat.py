"""The partial sums of a split row, read by the last chunk's whole warp: every pass over a
row of many chunks reads them all, so repeated solves give the same bits, and the row's
product equals a plain sum."""
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


# chunks of the dense row: one more than a warp has lanes, and many
@pytest.mark.parametrize("n", [33 * 512, 60001])
@pytest.mark.parametrize("precision", [0, 1])
def test_split_sums_repeat(lpm, n, precision):
    data = lpgen.with_dense_lines(lpgen.large_mixed(7, m=2000, n=n - 1), seed=1)
    with lpm.LP(data, eta=0.9 / 300.0, check_every=16, max_iter=160, precision=precision) as g:
        assert g.info().n_split_slices >= n // 512
        runs = []
        for _ in range(20):
            g.set_state()
            assert g.solve(1e-300) == lpm.LP_ITER_LIMIT
            runs.append((g.state(), g.info()))
    want, info = runs[0]
    for got, _ in runs[1:]:
        for k in want:
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    # the residual of the average at the last check: each row of A x is off by at most
    # len(row) eps times the sum of its terms' sizes, in any order of summation
    x = want["xbar"]
    prod = data.val * x[data.col_idx]
    rows = np.repeat(np.arange(data.m), np.diff(data.row_ptr))
    ax = np.bincount(rows, weights=prod, minlength=data.m)
    mag = np.bincount(rows, weights=np.abs(prod), minlength=data.m)
    v = data.b - ax
    v = np.where(data.row_type == lpgen.ROW_EQ, v,
                 np.where(data.row_type == lpgen.ROW_GE, np.maximum(v, 0.0), np.minimum(v, 0.0)))
    rounding = 2.0 ** -51 * np.diff(data.row_ptr) * mag  # of both sides
    assert abs(info.kkt_avg[0] - np.linalg.norm(v)) <= np.linalg.norm(rounding) + 1e-13 * np.linalg.norm(v)
