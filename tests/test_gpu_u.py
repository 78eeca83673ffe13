"""compute_U in closed form against the oracle at the edges of its dispatch:
FP64 above the orders the other tests cover, the mixed path on both sides of the
order where the layer recursion gives way to it, a block of 32 atoms that is not
full, neighbour counts that differ between its atoms, and the same pairs handed
over as a caller's list."""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.parity_util import rel_err
from tests.test_gpu_parity import FP64_TOL, full_check, snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def ragged(seed):
    cfg = inputs.bcc(3, disp=0.2, seed=seed)
    return inputs.Config(pos=np.ascontiguousarray(cfg.pos[:53]), box=cfg.box, name="bcc3 less one")


@pytest.mark.parametrize("twojmax,prec", [(9, 0), (11, 0), (13, 0), (9, 1), (10, 1), (13, 1)])
def test_orders_and_ragged_blocks(snapmod, twojmax, prec):  # noqa: F811
    full_check(snapmod, twojmax, ragged(61 + twojmax), prec)


@pytest.mark.parametrize("twojmax,prec", [(8, 0), (9, 1), (10, 1)])
def test_caller_list_gives_the_same_u(snapmod, twojmax, prec):  # noqa: F811
    """The internal list handed back by the caller: the slots keep their order,
    so U is the same but for the geometry's evaluation in another kernel."""
    cfg = ragged(80 + twojmax)
    s = snapmod.Snap(twojmax, inputs.beta(twojmax), precision=prec)
    pos = torch.tensor(cfg.pos, dtype=torch.float64, device="cuda:0")
    s.compute(pos, cfg.box)
    n = cfg.natoms
    K = s.get_buffer(snapmod.BUF_NBR_IDX).size // n
    cnt, idx, img = [s.get_buffer(b).copy() for b in
                     (snapmod.BUF_NBR_CNT, snapmod.BUF_NBR_IDX, snapmod.BUF_NBR_IMG)]
    U0 = s.get_buffer(snapmod.BUF_ULISTTOT).copy()
    dev = [torch.tensor(x, device="cuda:0") for x in (cnt.astype(np.int32), idx.reshape(n, K).astype(np.int32),
                                                      img.reshape(n, K, 3).astype(np.int8))]
    s.compute(pos, cfg.box, neighbors=tuple(dev))
    U1 = s.get_buffer(snapmod.BUF_ULISTTOT).copy()
    s.close()
    assert rel_err(U1, U0) <= (FP64_TOL if prec == 0 else 1e-6)
