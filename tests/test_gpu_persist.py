"""The persistent compute_Y where a CTA takes several items, so that it stages a
block over the one before: the same bits as the default launch.  16000 atoms are
1000 blocks of 16 atoms in FP64 and 500 of 32 in mixed precision, before any is
split, on at most two resident CTAs an SM."""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,twojmax", [(0, 2), (0, 8), (0, 14), (1, 8), (1, 14)])
def test_items_taken_one_after_the_other_change_no_bit(snapmod, prec, twojmax):  # noqa: F811
    cfg = inputs.bcc(20, disp=0.15, seed=91)
    s = snapmod.Snap(twojmax, inputs.beta(twojmax), precision=prec)
    pos = torch.tensor(cfg.pos, device="cuda:0")
    ref = [x.cpu().numpy().copy() for x in s.compute(pos, cfg.box)]
    y = s.get_buffer(snapmod.BUF_YLIST).copy()
    s.set_knob(snapmod.KNOB_PERSIST, 1)
    for _ in range(3):
        for a, b in zip(s.compute(pos, cfg.box), ref):
            assert np.array_equal(a.cpu().numpy(), b)
        assert np.array_equal(s.get_buffer(snapmod.BUF_YLIST), y)
    s.close()
