"""The choice between clusters and the per-pass kernels counts how many clusters fit at
once: batches whose clusters would run one round after the other are not slower than with
the per-pass kernels (autotune = 0), and batches of small problems keep their clusters."""
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


def ms_per_block(lpm, probs, autotune, precision):
    import torch

    with lpm.LPBatch(probs, eta=0.01, check_every=64, precision=precision, autotune=autotune,
                     tuning={"autotune": 1, "max_k_shift": 0}) as g:
        g.iterate(2, 1e-300)
        best = np.inf
        for _ in range(5):
            torch.cuda.synchronize()
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            g.iterate(4, 1e-300)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1) / 4)
    return best


# clusters of 8 with one block per SM fit 15 times; measured with clusters / per-pass
# kernels, us per iteration: 27.7 / 12.3, 26.1 / 13.0, 41.8 / 33.5 -- and 3.6 / 11.1, 5.6 / 8.9
@pytest.mark.parametrize("count,m,n,precision,limit", [
    (16, 4000, 8000, 0, 1.2), (16, 2000, 4000, 1, 1.2), (128, 2000, 4000, 0, 1.2),
    (64, 200, 400, 0, 0.7), (64, 200, 400, 1, 0.85)])
def test_not_slower_than_the_per_pass_kernels(lpm, count, m, n, precision, limit):
    base = [lpgen.tiny_standard_form(k, m=m, n=n) for k in range(3)]
    probs = [base[k % 3] for k in range(count)]
    assert ms_per_block(lpm, probs, 1, precision) < limit * ms_per_block(lpm, probs, 0, precision)
