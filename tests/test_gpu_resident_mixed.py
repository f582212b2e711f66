"""Mixed precision, single LPs, every restart scheme: the resident kernels (one cluster, the
grid with two blocks per SM, the whole grid) form the radius of either candidate in the order
of the per-pass kernels, so the corrections that it scales, and the iterates, are the same bit
for bit."""
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


SIZES = [(200, 500), (997, 4999), (5000, 25000), (12000, 60000)]


@pytest.mark.parametrize("m,n", SIZES)
@pytest.mark.parametrize("scheme", ["NONE", "FIXED", "ADAPTIVE", "FLEXIBLE"])
def test_schemes(lpm, m, n, scheme):
    data = lpgen.large_mixed(6, m=m, n=n)
    out = []
    for autotune in (1, 0):
        with lpm.LP(data, eta=0.05, omega=0.25, check_every=16, max_iter=16 * 20, fixed_len=48,
                    precision=1, autotune=autotune,
                    restart_scheme=getattr(lpm, "LP_RESTART_" + scheme)) as g:
            status = g.solve(1e-300)
            info = g.info()
            assert (info.graph_kernels == 1) == bool(autotune)
            out.append((status, info.restarts, g.state(), g.trace()))
    assert out[0][:2] == out[1][:2]
    if scheme in ("FIXED", "ADAPTIVE", "FLEXIBLE"):
        assert out[0][1] > 0
    for k in out[0][2]:
        np.testing.assert_array_equal(out[0][2][k], out[1][2][k], err_msg=k)
    np.testing.assert_array_equal(out[0][3][:, [0, 2]], out[1][3][:, [0, 2]])
