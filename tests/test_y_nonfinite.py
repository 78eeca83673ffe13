"""A coefficient that is not finite reaches every output of compute_Y that
depends on it, in the class stream's FP32 form and in its fixed point, whatever
other coefficients follow it in the stream (host walk, no GPU)."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("twojmax", [0, 1, 4, 8])
def test_every_dependent_output(snapmod, precision, twojmax):
    n = snapmod.num_coeff(twojmax)
    h = symmetric_u(snapmod, twojmax, np.random.default_rng(7))
    good = inputs.beta(twojmax)
    for comp in range(1, n + 1):
        # Y is linear in beta: the outputs of this component alone
        unit = np.zeros(n + 1)
        unit[comp] = 1.0
        depends = np.abs(snapmod.yi_host(twojmax, unit, h, precision=1)).max(axis=-1) > 0
        assert depends.any()
        for bad in (np.nan, np.inf, -np.inf):
            beta = good.copy()
            beta[comp] = bad
            y = snapmod.yi_host(twojmax, beta, h, precision=precision)
            finite = np.isfinite(y).all(axis=-1)
            assert not finite[depends].any(), (comp, bad)
            assert finite[~depends].all(), (comp, bad)
