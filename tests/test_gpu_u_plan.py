"""compute_U's split into CTAs: whatever it is, the same bits.  An atom's U does not
depend on the atoms around its block, so the first atoms of a long list of
configurations have the U that they have alone, where blocks are few and every
unit has a CTA of its own."""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("twojmax,prec", [(0, 0), (1, 0), (2, 0), (3, 0), (4, 0), (5, 0), (6, 0), (7, 0), (8, 0), (11, 0),
                                          (14, 0), (0, 1), (5, 1), (10, 1), (14, 1)])
def test_any_split_gives_the_same_u(snapmod, twojmax, prec):  # noqa: F811
    one = inputs.bcc(2, disp=0.1, seed=5)
    s = snapmod.Snap(twojmax, inputs.beta(twojmax), precision=prec)
    H = snapmod.half_size(twojmax)
    s.compute(torch.tensor(one.pos, device="cuda:0"), one.box)
    want = s.get_buffer(snapmod.BUF_ULISTTOT).reshape(-1, H, 2).copy()
    for copies in (3, 20, 150, 600):  # 48 to 9600 atoms: splits from a unit a CTA to nine
        cfgs = [one] * copies
        pos = torch.tensor(np.concatenate([c.pos for c in cfgs]), device="cuda:0")
        s.compute_batch(pos, np.array([c.natoms for c in cfgs]), np.array([c.box for c in cfgs]))
        got = s.get_buffer(snapmod.BUF_ULISTTOT).reshape(copies, one.natoms, H, 2)
        assert all(np.array_equal(g, want) for g in got), copies
    s.close()
