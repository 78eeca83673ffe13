"""snap_set_beta: whatever order it and the choice of compute_Y's layout come in,
and whatever was evaluated or captured before, the step is bit for bit that of a
context made with the new coefficients."""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("twojmax", [0, 1, 5, 8, 14])
def test_new_coefficients(snapmod, prec, twojmax):  # noqa: F811
    cfg = inputs.bcc(3, disp=0.1, seed=23)
    pos = torch.tensor(cfg.pos, device="cuda:0")
    old, new = inputs.beta(twojmax, seed=3), inputs.beta(twojmax, seed=4)

    def step(s):
        return [x.cpu().numpy().copy() for x in s.compute(pos, cfg.box)]

    want = []
    for layout in (0, 1):
        s = snapmod.Snap(twojmax, new, precision=prec)
        s.set_knob(snapmod.KNOB_YI_LAYOUT, layout)
        want.append(step(s))
        s.close()
    same = lambda a, b: all(np.array_equal(x, y) for x, y in zip(a, b))  # noqa: E731
    s = snapmod.Snap(twojmax, old, precision=prec)
    first = step(s)
    assert not same(first, want[0])
    s.set_beta(new)
    assert same(step(s), want[0])
    s.set_knob(snapmod.KNOB_YI_LAYOUT, 1)  # the list of terms is made here
    assert same(step(s), want[1])
    s.set_beta(old)
    step(s)
    s.set_knob(snapmod.KNOB_YI_LAYOUT, 0)
    assert same(step(s), first)
    s.set_beta(new)
    assert same(step(s), want[0])
    s.set_knob(snapmod.KNOB_YI_LAYOUT, 1)
    assert same(step(s), want[1])
    s.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_coefficients_that_are_not_finite(snapmod, prec):  # noqa: F811
    """They reach every atom's energy and force, and leave with the next beta."""
    cfg = inputs.bcc(3, disp=0.1, seed=23)
    pos = torch.tensor(cfg.pos, device="cuda:0")
    beta = inputs.beta(4)
    s = snapmod.Snap(4, beta, precision=prec)
    ref = [x.cpu().numpy().copy() for x in s.compute(pos, cfg.box)]
    for bad in (np.nan, np.inf):
        for comp in range(1, len(beta)):
            b = beta.copy()
            b[comp] = bad
            s.set_beta(b)
            e, f, _ = [x.cpu().numpy() for x in s.compute(pos, cfg.box)]
            assert not np.isfinite(e).any() and not np.isfinite(f).all(axis=1).any(), (comp, bad)
    s.set_beta(beta)
    assert all(np.array_equal(x.cpu().numpy(), y) for x, y in zip(s.compute(pos, cfg.box), ref))
    s.close()
