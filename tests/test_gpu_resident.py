"""The resident kernel (autotune = 1, LPs that fit on the SMs) against the
per-pass kernels (autotune = 0): the same lanes, chains and butterflies (and, in
mixed precision, the same order of the radius that scales the next correction),
so the iterates agree bit for bit; the check's other sums are reduced in another
order, so its gaps and residuals agree to rounding and the restart decisions are
equal."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2105_12715_gb300 import lpgen  # noqa: E402


@pytest.fixture(scope="module")
def lpm():
    from paper_2105_12715_gb300 import lp
    return lp


def without_rows(n):
    d = lpgen.tiny_standard_form(1, m=1, n=n, per_col=1)
    return dataclasses.replace(d, m=0, row_ptr=np.zeros(1, np.int32), col_idx=np.zeros(0, np.int32),
                               val=np.zeros(0), b=np.zeros(0), row_type=np.zeros(0, np.int8),
                               ub=np.ones(n), c=np.linspace(-1.0, 1.0, n))


CASES = {  # one slice; 4, 5 and 17 slices per block's share; ragged tails; empty rows and columns
    "1x1": lambda: lpgen.tiny_standard_form(0, m=1, n=1, per_col=1),
    "no_rows": lambda: without_rows(33),
    "31x33": lambda: lpgen.tiny_standard_form(1, m=31, n=33, per_col=3),
    "200x400": lambda: lpgen.tiny_standard_form(0),
    "empty_lines": lambda: lpgen.adversarial(7),
    "dense_lines": lambda: lpgen.adversarial(9, m=400, n=450),
    "997x4999": lambda: lpgen.large_mixed(3, m=997, n=4999),
    "5000x25000": lambda: lpgen.large_mixed(4, m=5000, n=25000),
    "20000x90001": lambda: lpgen.large_mixed(5, m=20000, n=90001),
}


def run(lpm, data, autotune, **opts):
    with lpm.LP(data, eta=0.05, autotune=autotune, **opts) as g:
        status = g.solve(1e-300)
        return status, g.state(), g.trace(64), g.info()


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("precision", [0, 1])
def test_same_iterates_as_the_per_pass_kernels(lpm, name, precision):
    data = CASES[name]()
    opts = dict(check_every=24, max_iter=24 * 6 + 7, precision=precision)  # and a partial block
    s1, a, t1, i1 = run(lpm, data, 1, **opts)
    s0, b, t0, i0 = run(lpm, data, 0, **opts)
    assert i1.graph_kernels == 1 and i0.graph_kernels > 48
    assert (s1, i1.iters, i1.restarts, i1.returned) == (s0, i0.iters, i0.restarts, i0.returned)
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    np.testing.assert_array_equal(t1[:, [0, 2]], t0[:, [0, 2]])
    if precision == 0:
        # a gap sums n + m positive terms in another order: n eps relative, and residuals
        # of size |b| cancel down to the KKT error
        np.testing.assert_allclose(t1[:, [1, 3, 4, 5]], t0[:, [1, 3, 4, 5]], rtol=1e-9, atol=1e-11)


@pytest.mark.parametrize("scheme", ["NONE", "FIXED", "FLEXIBLE"])
def test_schemes(lpm, scheme):
    data = lpgen.large_mixed(6, m=700, n=3100)
    opts = dict(check_every=16, max_iter=16 * 20, fixed_len=48, omega=0.25,
                restart_scheme=getattr(lpm, "LP_RESTART_" + scheme))
    s1, a, t1, i1 = run(lpm, data, 1, **opts)
    s0, b, t0, i0 = run(lpm, data, 0, **opts)
    assert i1.graph_kernels == 1 and (s1, i1.restarts) == (s0, i0.restarts)
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    np.testing.assert_allclose(t1, t0, rtol=1e-9, atol=1e-11)


def test_check_periods_at_the_edge(lpm):
    """K = 1 and K = 1024 run resident; K = 1025 exceeds the weights' space."""
    data = lpgen.tiny_standard_form(2)
    for k, resident in ((1, True), (1024, True), (1025, False)):
        _, a, _, i1 = run(lpm, data, 1, check_every=k, max_iter=2 * k)
        _, b, _, _ = run(lpm, data, 0, check_every=k, max_iter=2 * k)
        assert (i1.graph_kernels == 1) == resident
        for key in a:
            np.testing.assert_array_equal(a[key], b[key], err_msg=f"{k} {key}")


def test_converges_and_repeats(lpm):
    """Solves to 1e-8, twice from the same start on one handle: same bits."""
    data = lpgen.large_mixed(11, m=300, n=1500)
    with lpm.LP(data, omega=0.0625, max_iter=400000) as g:
        outs = []
        for _ in range(2):
            g.set_state()
            assert g.solve(1e-8) == lpm.LP_OK
            outs.append(g.solution() + (g.info().iters,))
        assert g.info().graph_kernels == 1
    assert outs[0][2] == outs[1][2]
    np.testing.assert_array_equal(outs[0][0], outs[1][0])
    np.testing.assert_array_equal(outs[0][1], outs[1][1])
    assert abs(np.dot(data.c, outs[0][0]) - data.obj_star) <= 1e-6 * (1 + abs(data.obj_star))


def batch_run(lpm, probs, autotune, **opts):
    with lpm.LPBatch(probs, autotune=autotune, eta=0.05, **opts) as g:
        status = g.solve(1e-300)
        return status, g.state(), g.info()[1]


BATCHES = {  # clusters of 8, 2 and 1 blocks, matrix inside; streamed, several blocks per SM
    "3_uneven": lambda: [lpgen.tiny_standard_form(1, m=31, n=33, per_col=3), lpgen.adversarial(7),
                         lpgen.large_mixed(3, m=199, n=701)],
    "70": lambda: [lpgen.tiny_standard_form(k, m=90 + k, n=200, per_col=4) for k in range(70)],
    "160": lambda: [lpgen.adversarial(k, m=20 + k % 7, n=41) for k in range(160)],
    "640": lambda: [lpgen.tiny_standard_form(k, m=60, n=121, per_col=4) for k in range(640)],
}


@pytest.mark.parametrize("name", list(BATCHES))
@pytest.mark.parametrize("precision", [0, 1])
def test_batch_same_iterates_as_the_per_pass_kernels(lpm, name, precision):
    probs = BATCHES[name]()
    opts = dict(check_every=16, max_iter=16 * 9, precision=precision)
    s1, a, p1 = batch_run(lpm, probs, 1, **opts)
    s0, b, p0 = batch_run(lpm, probs, 0, **opts)
    assert s1 == s0
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    for u, v in zip(p1, p0):
        for k in ("iters", "restarts", "checks", "status", "returned"):
            assert u[k] == v[k], k
        if precision == 0:
            np.testing.assert_allclose(u["kkt_avg"], v["kkt_avg"], rtol=1e-9, atol=1e-11)
            np.testing.assert_allclose(u["rho_stored"], v["rho_stored"], rtol=1e-9, atol=1e-11)


def test_batch_check_periods_and_schemes(lpm):
    """Problems due at different blocks, flexible and fixed restarts, and an
    iteration limit that falls between two checks."""
    probs = [lpgen.large_mixed(k, m=120 + 10 * k, n=400) for k in range(5)]
    for scheme in ("FLEXIBLE", "FIXED", "NONE"):
        got = []
        for autotune in (1, 0):
            with lpm.LPBatch(probs, autotune=autotune, eta=0.05, check_every=16, fixed_len=48,
                             max_iter=16 * 11,
                             restart_scheme=getattr(lpm, "LP_RESTART_" + scheme)) as g:
                g.set_check_every([16, 32, 48, 64, 16])
                g.solve(1e-300)
                got.append((g.state(), g.info()[1]))
        for k in got[0][0]:
            np.testing.assert_array_equal(got[0][0][k], got[1][0][k], err_msg=f"{scheme} {k}")
        for u, v in zip(got[0][1], got[1][1]):
            for k in ("iters", "restarts", "checks", "status", "returned"):
                assert u[k] == v[k], (scheme, k)


@pytest.mark.parametrize("name", ["31x33", "200x400", "empty_lines", "997x4999"])
def test_adjoint_is_the_per_pass_adjoint(lpm, name):
    """One launch for the whole reverse sweep against the launches pass by pass:
    the same recurrence with the same sums; only c and b's gradients and the state
    left behind come back."""
    data = CASES[name]()
    rng = np.random.default_rng(5)
    wx, wy = rng.standard_normal(data.n), rng.standard_normal(data.m)
    out = []
    for autotune in (1, 0):
        with lpm.LP(data, eta=0.05, autotune=autotune, check_every=20) as g:
            lpm.lp_solve_recorded(g.h, 100)
            before = g.state()
            dc, db = np.empty(data.n), np.empty(data.m)
            for _ in range(2):  # a second call repeats the first
                lpm.lp_backward(g.h, wx, wy, dc, db)
            after = g.state()
            for k in before:
                np.testing.assert_array_equal(after[k], before[k], err_msg=k)
            out.append((dc, db, g.info().graph_kernels))
    assert out[0][2] == 1 and out[1][2] > 1
    # per-pass launches contract the recurrence's products into FMAs differently
    for a, b in zip(out[0][:2], out[1][:2]):
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-12 * max(1.0, np.abs(b).max(initial=0.0)))


def test_batch_adjoint_is_the_per_pass_adjoint(lpm):
    for probs in (BATCHES["3_uneven"](), BATCHES["640"]()):
        n, m = sum(p.n for p in probs), sum(p.m for p in probs)
        rng = np.random.default_rng(6)
        wx, wy = rng.standard_normal(n), rng.standard_normal(m)
        out = []
        for autotune in (1, 0):
            with lpm.LPBatch(probs, eta=0.05, autotune=autotune, check_every=16) as g:
                g.solve_recorded(80)
                before = g.state()
                out.append(g.backward(wx, wy))
                after = g.state()
                for k in before:
                    np.testing.assert_array_equal(after[k], before[k], err_msg=k)
        for a, b in zip(*out):
            np.testing.assert_allclose(a, b, rtol=0, atol=1e-12 * max(1.0, np.abs(b).max()))


@pytest.mark.parametrize("name", ["1x1", "no_rows", "empty_lines", "997x4999", "20000x90001"])
@pytest.mark.parametrize("scheme,precision", [("ADAPTIVE", 0), ("FLEXIBLE", 0), ("ADAPTIVE", 1)])
def test_search_by_newton_steps_in_the_per_pass_check(lpm, name, scheme, precision):
    """K = 1025 exceeds the resident kernels: one search launch against the radix
    passes.  Both sum n + m positive terms and take one square root."""
    data = CASES[name]()
    opts = dict(check_every=1025, max_iter=2050, precision=precision,
                restart_scheme=getattr(lpm, "LP_RESTART_" + scheme))
    _, a, t1, i1 = run(lpm, data, 1, **opts)
    _, b, t0, i0 = run(lpm, data, 0, **opts)
    assert i1.graph_kernels == i0.graph_kernels - 15
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    np.testing.assert_allclose(t1, t0, rtol=1e-9, atol=1e-11)


@pytest.mark.parametrize("scheme", ["ADAPTIVE", "FLEXIBLE"])
def test_batch_search_at_the_edges_of_its_cluster(lpm, scheme):
    """n + m = 2047 (one block), 2048 and more (a cluster), against single solves."""
    sizes = [(1, 1), (447, 1600), (448, 1600), (449, 1600), (3000, 9001), (255, 1)]
    probs = [lpgen.tiny_standard_form(k, m=m, n=n, per_col=min(m, 4))
             for k, (m, n) in enumerate(sizes)]
    opts = dict(check_every=16, max_iter=16, restart_scheme=getattr(lpm, "LP_RESTART_" + scheme))
    _, _, infos = batch_run(lpm, probs, 0, **opts)
    for p, u in zip(probs, infos):
        _, _, _, i = run(lpm, p, 0, **opts)
        # the iterates of 16 steps agree to rounding, so do the gaps
        np.testing.assert_allclose(u["last_rho"], i.last_rho, rtol=1e-9, atol=1e-11)
