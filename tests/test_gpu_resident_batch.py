"""Batches in clusters of 1, 2, 4 and 8 blocks, matrix inside and streamed, under the
adaptive and the flexible scheme, against the per-pass kernels (autotune = 0): the same
iterates bit for bit, on every repeat.

Among them problems whose first check restarts without a step of the multiplier
search (every coordinate's full move to its bound lies inside the trust region): no
barrier follows the check's there, so no block may still need another block's rows."""
import ctypes as C
import dataclasses

import numpy as np
import pytest

from paper_2105_12715_gb300 import lpgen

ETA, K = 0.05, 16


def box_with_slack_rows(seed, m, n, rows=True):
    """min c x, 0 <= x <= 1, rows that never bind.  Nine columns of ten reach their
    bound within K steps, the others creep, so the LP is not solved at the first check."""
    d = lpgen.tiny_standard_form(seed, m=m, n=n, per_col=4)
    rng = np.random.default_rng(1000 + seed)
    slow = np.arange(n) % 10 == 3
    c = -np.where(slow, rng.uniform(0.05, 0.2, n), rng.uniform(3.0, 8.0, n))
    sense = np.where(np.arange(m) % 2 == 0, lpgen.ROW_GE, lpgen.ROW_LE).astype(np.int8)
    d = dataclasses.replace(d, c=c, ub=np.ones(n), row_type=sense,
                            b=np.where(sense == lpgen.ROW_GE, -1e3, 1e3))
    if rows:
        return d
    return dataclasses.replace(d, m=0, row_ptr=np.zeros(1, np.int32), col_idx=np.zeros(0, np.int32),
                               val=np.zeros(0), b=np.zeros(0), row_type=np.zeros(0, np.int8))


def test_the_first_check_needs_no_search_step():
    """Of both candidates: no coordinate may move without bound, and the move of all of
    them to their bounds is inside the ball around the start (omega = 1)."""
    d = box_with_slack_rows(0, 300, 700)
    A = np.zeros((d.m, d.n))
    for i in range(d.m):
        A[i, d.col_idx[d.row_ptr[i]:d.row_ptr[i + 1]]] = d.val[d.row_ptr[i]:d.row_ptr[i + 1]]
    x, xbar, y = np.zeros(d.n), np.zeros(d.n), np.zeros(d.m)
    for k in range(K):
        xn = np.clip(x - ETA * (d.c - A.T @ y), 0.0, 1.0)
        y = y - ETA * (A @ (2 * xn - x) - d.b)
        y = np.where(d.row_type == lpgen.ROW_GE, np.maximum(y, 0.0), np.minimum(y, 0.0))
        x, xbar = xn, xbar + (xn - xbar) / (k + 1)
    assert not y.any()  # every row is slack and its multiplier sits at its bound
    for z in (xbar, x):
        assert 0.0 < np.sum((1.0 - z) ** 2) < np.sum(z ** 2)


@pytest.fixture(scope="module")
def lpm():
    import torch

    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2105_12715_gb300 import lp

    lp.load()
    return lp


def sms():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


def box_mix(count):
    return [box_with_slack_rows(k, 300 + k % 5, 700, rows=k % 4 != 3) for k in range(count)]


def uneven(count, m, n):
    return [lpgen.large_mixed(k, m=m + k % 7, n=n) for k in range(count)]


# batches that give a problem 8, 4, 2 and 1 blocks, the matrix inside or streamed (the
# shapes that test_shapes_covered expects at 152 SMs)
BATCHES = {
    "box, 19": lambda: box_mix(19),
    "box, 50": lambda: box_mix(50),
    "box, 101": lambda: box_mix(101),
    "box, 160": lambda: box_mix(160),
    "mixed rows, 101": lambda: uneven(101, 90, 200),
    "200 x 400, 330": lambda: [lpgen.tiny_standard_form(k % 5) for k in range(330)],
    "1000 x 2000, 101": lambda: [lpgen.tiny_standard_form(k % 3, m=1000, n=2000)
                                 for k in range(101)],
    "1400 x 2800, 40": lambda: [lpgen.tiny_standard_form(k % 3, m=1400, n=2800)
                                for k in range(40)],
}


def shape(lpm, g):
    f, b = C.c_int32(), C.c_int32()
    assert lpm.load().lp_batch_shape(g.h, C.byref(f), C.byref(b)) == lpm.LP_OK
    return f.value


@pytest.mark.gpu
def test_shapes_covered(lpm):
    """Negative: the matrix is streamed."""
    if sms() != 152:
        pytest.skip("the choice depends on the number of SMs")
    seen = {0: set(), 1: set()}
    for precision in seen:
        for make in BATCHES.values():
            with lpm.LPBatch(make(), eta=ETA, check_every=K, precision=precision) as g:
                seen[precision].add(shape(lpm, g))
    for precision, got in seen.items():
        assert {8, 4} <= got and {1, 2, -1, -2} & got and {-8, -4, -2} & got, (precision, got)


@pytest.mark.gpu
@pytest.mark.parametrize("name", list(BATCHES))
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("scheme", ["ADAPTIVE", "FLEXIBLE"])
def test_batch_iterates_repeat_and_equal_the_per_pass_kernels(lpm, name, precision, scheme):
    probs = BATCHES[name]()
    opts = dict(eta=ETA, check_every=K, max_iter=5 * K, precision=precision,
                restart_scheme=getattr(lpm, "LP_RESTART_" + scheme))
    with lpm.LPBatch(probs, autotune=0, **opts) as g:
        want_status = g.solve(1e-300)
        want, infos = g.state(), g.info()[1]
    with lpm.LPBatch(probs, autotune=1, **opts) as g:
        for _ in range(12):
            g.set_state()
            assert g.solve(1e-300) == want_status
            got = g.state()
            for k in want:
                np.testing.assert_array_equal(got[k], want[k], err_msg=k)
            for u, v in zip(g.info()[1], infos):
                for k in ("iters", "restarts", "checks", "status", "returned"):
                    assert u[k] == v[k], k
