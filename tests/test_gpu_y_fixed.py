"""FP64 compute_Y where an atom's U spans many powers of two: pairs just inside the
cutoff, whose f_c is 2^-20 to 2^-44, beside close ones.  On the device against the
host walk of the same fixed point, and the whole step against the oracle."""
import numpy as np
import pytest

from oracle import snap_oracle as O
from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RCUT = inputs.RCUT


def faint_pairs():
    """Dimers and one chain in a wide box, in directions of no symmetry."""
    rng = np.random.Generator(np.random.PCG64(5))
    pos = []
    for k, delta in enumerate((3e-3, 2e-4, 1e-5, 8e-7)):
        d = rng.normal(size=3)
        c = np.array([12.0 * k + 6.0, 8.0, 9.0])
        pos += [c, c + d / np.linalg.norm(d) * (RCUT - delta)]
    d, f = rng.normal(size=3), rng.normal(size=3)
    c = np.array([8.0, 30.0, 30.0])
    pos += [c, c + d / np.linalg.norm(d) * 2.6, c - d / np.linalg.norm(d) * (RCUT - 1e-5) + 1e-7 * f]
    return inputs.Config(pos=np.array(pos), box=np.array([60.0, 45.0, 45.0]), name="faint pairs")


@pytest.mark.parametrize("twojmax", [1, 4, 8, 11, 14])
def test_device_walks_the_same_fixed_point(snapmod, twojmax):  # noqa: F811
    cfg = faint_pairs()
    beta = inputs.beta(twojmax)
    s = snapmod.Snap(twojmax, beta, precision=0)
    s.compute(torch.tensor(cfg.pos, device="cuda:0"), cfg.box)
    H, n = snapmod.half_size(twojmax), cfg.natoms
    U = s.get_buffer(snapmod.BUF_ULISTTOT).reshape(n, H, 2)
    Y = s.get_buffer(snapmod.BUF_YLIST).reshape(n, H, 2)
    s.close()
    spread = np.abs(U[np.abs(U) > 0])
    assert spread.max() / spread.min() > 2.0 ** 40
    read = [snapmod.half_index(twojmax, t, ma, mb) for t in range(twojmax + 1) for mb in range(t // 2 + 1)
            for ma in range(t + 1) if not (2 * mb == t and ma > mb)]
    for i in range(n):
        want = snapmod.yi_host(twojmax, beta, U[i], precision=0)[read]
        got = Y[i][read]
        # the sums are the same whole numbers; they are turned into FP64 (and the
        # two halves of a split one added) with a few roundings
        top = np.abs(want).max()
        ok = np.abs(got - want) <= 2.0 ** -45 * np.abs(want) + 2.0 ** -64 * top
        assert ok.all(), (i, np.abs(got - want)[~ok], want[~ok])


@pytest.mark.parametrize("twojmax", [4, 8, 14])
def test_faint_forces(snapmod, twojmax):  # noqa: F811
    """Each atom's force relative to its own size.  f_c is sin^2 of (rcut - r) in
    units of the span, so r, rounded at 2^-53 of 5 A, is known to 1e-9 of the
    smallest rcut - r; ten such roundings are allowed."""
    cfg = faint_pairs()
    beta = inputs.beta(twojmax)
    _, ref = O.evaluate(O.Params(twojmax), beta, cfg.pos, cfg.box)
    s = snapmod.Snap(twojmax, beta, precision=0)
    e, f, _ = [x.cpu().numpy() for x in s.compute(torch.tensor(cfg.pos, device="cuda:0"), cfg.box)]
    s.close()
    size = np.linalg.norm(ref.F, axis=1)
    assert size.min() > 0 and size.max() / size.min() > 1e3
    assert (np.linalg.norm(f - ref.F, axis=1) <= 1e-8 * size).all()
    assert np.abs(e - ref.E).max() <= 1e-12 * np.abs(ref.E).max()
