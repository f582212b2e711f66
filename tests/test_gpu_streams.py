"""Several LPs at once, each with its own handle and stream: the results are those of each
alone, and LPs that leave half of the GPU idle share it."""
import dataclasses
import threading

import numpy as np
import pytest

from paper_2105_12715_gb300 import lpgen

pytestmark = pytest.mark.gpu

K = 64


@pytest.fixture(scope="module")
def lpm():
    import torch

    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2105_12715_gb300 import lp

    lp.load()
    return lp


# one cluster; the grid with room for two blocks per SM, FP64 and mixed; the whole grid;
# per-pass kernels with the search in one launch (K > 1024)
MIX = [dict(m=200, n=500), dict(m=997, n=4999), dict(m=1500, n=6000),
       dict(m=997, n=4999, precision=1), dict(m=5000, n=25000, precision=1),
       dict(m=5000, n=25000), dict(m=2000, n=9000, check_every=1025)]


def make(lpm, spec, stream):
    spec = {"check_every": K, "max_iter": 3 * 1025, **spec}
    data = lpgen.large_mixed(3, m=spec.pop("m"), n=spec.pop("n"))
    return lpm.LP(data, eta=0.05, stream=stream, **spec)


def test_results_of_handles_on_their_own_streams(lpm):
    import torch

    alone = []
    for spec in MIX:
        with make(lpm, spec, torch.cuda.Stream()) as g:
            g.solve(1e-300)
            alone.append(g.state())
    handles = [make(lpm, spec, torch.cuda.Stream()) for spec in MIX]
    try:
        for _ in range(3):
            for g in handles:
                g.set_state()
            threads = [threading.Thread(target=g.solve, args=(1e-300,)) for g in handles]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            for g, want in zip(handles, alone):
                assert g.info().iters == 3 * 1025
                got = g.state()
                for k in want:
                    np.testing.assert_array_equal(got[k], want[k], err_msg=k)
    finally:
        for g in handles:
            g.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_four_lps_share_the_gpu(lpm, precision):
    """Four LPs of 2k x 10k on four streams take less than three times one of them (one
    after the other: four times; two at once: 2.3 times)."""
    import torch

    data = [lpgen.large_mixed(k, m=2000, n=10000) for k in range(4)]
    handles = [lpm.LP(d, eta=0.05, check_every=K, precision=precision, stream=torch.cuda.Stream())
               for d in data]

    def ms(some):
        best = np.inf
        for _ in range(6):
            torch.cuda.synchronize()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(1 + len(some))]
            e[0].record(some[0].stream)
            for g in some[1:]:
                g.stream.wait_event(e[0])
            for g in some:
                g.iterate(16, 1e-300)
            for g, end in zip(some, e[1:]):
                end.record(g.stream)
            torch.cuda.synchronize()
            best = min(best, max(e[0].elapsed_time(end) for end in e[1:]))
        return best

    try:
        ms(handles)
        assert ms(handles) < 3.0 * ms(handles[:1])
    finally:
        for g in handles:
            g.close()


def test_matrix_that_needs_more_blocks_than_its_slices(lpm):
    """Mixed precision, 1,200 dense rows of one slice each: 16 slices per block would not
    fit, four do.  The iterates are those of the per-pass kernels."""
    n = 1200
    rng = np.random.default_rng(0)
    data = dataclasses.replace(
        lpgen.tiny_standard_form(0, m=1, n=1, per_col=1), m=n, n=n,
        row_ptr=(np.arange(n + 1) * n).astype(np.int32),
        col_idx=np.tile(np.arange(n, dtype=np.int32), n), val=rng.standard_normal(n * n),
        c=rng.standard_normal(n), b=rng.standard_normal(n), lb=np.zeros(n), ub=np.full(n, np.inf),
        row_type=np.zeros(n, np.int8))
    out = []
    for autotune in (1, 0):
        with lpm.LP(data, eta=0.9 / 75.0, check_every=16, max_iter=80, precision=1,
                    split_row_len=0, autotune=autotune) as g:
            g.solve(1e-300)
            assert (g.info().graph_kernels == 1) == bool(autotune)
            out.append(g.state())
    for k in out[0]:
        np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=k)
