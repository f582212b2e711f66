"""The batch tuner times the kernels that run the batch: a class's cost per iteration, as
lp_batch_info reports it, against blocks of iterations timed from outside."""
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


def us_per_iteration(g, count):
    import torch

    g.set_check_every([K << 16] * count)  # no check is due
    g.iterate(4, 1e-300)
    best = np.inf
    for _ in range(8):
        torch.cuda.synchronize()
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        g.iterate(16, 1e-300)
        e1.record()
        e1.synchronize()
        best = min(best, 1e3 * e0.elapsed_time(e1) / (16 * K))
    return best


# 8 problems: two launches per iteration cost three times what the cluster kernel does
# per iteration, so a factor of two tells them apart and leaves room for the clock
@pytest.mark.parametrize("autotune", [1, 0], ids=["cluster", "per-pass"])
@pytest.mark.parametrize("precision", [0, 1])
def test_class_costs_are_those_of_the_kernels_that_run(lpm, autotune, precision):
    probs = [lpgen.tiny_standard_form(k, m=60, n=121, per_col=4) for k in range(8)]
    with lpm.LPBatch(probs, eta=0.05, check_every=K, autotune=autotune, precision=precision,
                     tuning={"autotune": 1, "max_k_shift": 2, "check_budget": 0.05}) as g:
        summary, per = g.info()
        measured = us_per_iteration(g, len(probs))
    cls = per[0]["size_class"]
    told, check = 1e3 * summary["class_iter_ms"][cls], 1e3 * summary["class_check_ms"][cls]
    assert 0.5 < told / measured < 2.0, (told, measured)
    # the smallest period whose check costs at most the budget of its iterations
    want = next((s for s in range(2) if check <= 0.05 * (K << s) * told), 2)
    assert summary["class_k"][cls] == K << want
