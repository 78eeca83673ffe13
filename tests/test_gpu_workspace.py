"""compute_Y's second halves share a buffer with the bispectrum derivative's
tangent: evaluations of the two kinds after one another give what each gives alone."""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("twojmax", [4, 8, 14])
def test_step_and_derivative_in_turn(snapmod, prec, twojmax):  # noqa: F811
    cfg = inputs.bcc(3, disp=0.1, seed=17)
    pos = torch.tensor(cfg.pos, device="cuda:0")
    g = torch.tensor(np.random.Generator(np.random.PCG64(3)).normal(size=cfg.pos.shape), device="cuda:0")
    beta = inputs.beta(twojmax)

    def step(s):
        return [x.cpu().numpy().copy() for x in s.compute(pos, cfg.box)]

    def deriv(s):
        return s.bispectrum_deriv(pos, cfg.box, g).cpu().numpy().copy()

    a, b = (snapmod.Snap(twojmax, beta, precision=prec) for _ in range(2))
    want, dwant = step(a), deriv(b)
    a.close()
    b.close()
    s = snapmod.Snap(twojmax, beta, precision=prec)
    for _ in range(3):
        assert np.array_equal(deriv(s), dwant)
        assert all(np.array_equal(x, y) for x, y in zip(step(s), want))
    s.close()
