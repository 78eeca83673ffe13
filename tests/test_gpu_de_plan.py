"""The fused dE where an SM holds a few batches, on both sides of the line from which
a batch is not shared any more: the same bits.  Per-pair dE/dr of copies of one
configuration, few enough to share and many enough not to."""
import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("twojmax", [1, 4, 8, 11, 14])
def test_sharing_by_size(snapmod, twojmax, prec):  # noqa: F811
    one = inputs.bcc(2, disp=0.1, seed=5)
    s = snapmod.Snap(twojmax, inputs.beta(twojmax), precision=prec)
    s.compute(torch.tensor(one.pos, device="cuda:0"), one.box)
    cnt = s.get_buffer(snapmod.BUF_NBR_CNT).copy()
    K = s.get_buffer(snapmod.BUF_NBR_IDX).size // one.natoms
    used = (np.arange(K)[None, :] < cnt[:, None]).ravel()
    want = s.get_buffer(snapmod.BUF_DEDR).reshape(-1, 3)[used].copy()
    # 16 atoms of about 26 neighbours: 13 batches a copy, 1 to 13 an SM of 152
    for copies in (12, 35, 46, 60, 90, 150):
        pos = torch.tensor(np.concatenate([one.pos] * copies), device="cuda:0")
        s.compute_batch(pos, np.array([one.natoms] * copies), np.array([one.box] * copies))
        got = s.get_buffer(snapmod.BUF_DEDR).reshape(copies, -1, 3)
        assert all(np.array_equal(g[used], want) for g in got), copies
    s.close()
