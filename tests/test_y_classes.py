"""compute_Y's class stream and its fixed-point form, on the host (no GPU).

snap_yi_host walks the stream the kernels walk: mixed precision with FP64
arithmetic in place of FP32, FP64 in the kernel's own fixed point (59-bit U,
60-bit coefficients, products without their lowest part).  The two must agree
to the fixed point's rounding at every order, for coefficients of any size and
spread, and a coefficient that is not finite must reach the outputs.
"""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_tables_host import symmetric_u


@pytest.fixture(scope="module")
def snapmod():
    from paper_2011_12875_gb300 import build, snap
    build.build()
    snap.load()
    return snap


# A product is rounded at 2^-59 of the largest |U| (1 here) times the largest sum
# of |c| over a record, a few times a row; an output has up to about 1000 rows,
# whose coefficients are at most that sum: 1000 x 4 x 2^-59 = 7e-15 of it.  The
# outputs are compared relative to their largest, which is above a hundredth of
# the largest sum, and the FP64 walk rounds at 2^-53 of each partial sum.
@pytest.mark.parametrize("twojmax", [0, 1, 3, 9, 14])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -900, 2.0 ** 900, "spread"])
def test_fixed_point_agrees_with_fp64(snapmod, twojmax, scale):
    rng = np.random.default_rng(31 + twojmax)
    h = symmetric_u(snapmod, twojmax, rng)
    beta = inputs.beta(twojmax, scale=1.0, seed=5)
    if scale == "spread":
        beta[1::2] *= 1e9
        beta[2::3] *= 1e-9
    else:
        beta *= scale
    fx = snapmod.yi_host(twojmax, beta, h, precision=0)
    fp = snapmod.yi_host(twojmax, beta, h, precision=1)
    assert np.isfinite(fx).all() and np.abs(fp).max() > 0
    assert np.abs(fx - fp).max() <= 1e-12 * np.abs(fp).max()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_coefficients_that_are_not_finite_reach_y(snapmod, precision, bad):
    h = symmetric_u(snapmod, 4, np.random.default_rng(3))
    beta = inputs.beta(4)
    beta[-1] = bad  # (4, 4, 4): every output of rank 4
    y = snapmod.yi_host(4, beta, h, precision=precision)
    assert not np.isfinite(y[snapmod.half_index(4, 4, 2, 2)]).all()
