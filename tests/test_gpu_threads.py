"""Two contexts of different orders on two host threads, each with its own stream:
every call launches and gives the bits it gives alone.  Their kernels are the same
functions with different shared memory, in calls that launch kernel by kernel
(the profiled step, the bispectrum)."""
import threading

import numpy as np
import pytest

from paper_2011_12875_gb300 import inputs
from tests.test_gpu_parity import snapmod  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,orders", [(0, (14, 10)), (0, (8, 6)), (1, (14, 11))])
def test_two_threads(snapmod, prec, orders):  # noqa: F811
    made = []
    for k, twojmax in enumerate(orders):
        cfg = inputs.bcc(2 + k, disp=0.1, seed=31 + k)
        s = snapmod.Snap(twojmax, inputs.beta(twojmax), precision=prec)
        pos = torch.tensor(cfg.pos, device="cuda:0")
        s.profile(True)
        ref = [x.cpu().numpy().copy() for x in s.compute(pos, cfg.box)] + [s.bispectrum(pos, cfg.box).cpu().numpy().copy()]
        made.append((s, pos, cfg.box, ref))
    torch.cuda.synchronize()
    start, wrong = threading.Barrier(2), []

    def work(s, pos, box, ref):
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            try:
                for _ in range(150):
                    got = [x.cpu().numpy() for x in s.compute(pos, box)] + [s.bispectrum(pos, box).cpu().numpy()]
                    if not all(np.array_equal(a, b) for a, b in zip(got, ref)):
                        wrong.append("bits")
            except Exception as e:  # noqa: BLE001
                wrong.append(repr(e))

    threads = [threading.Thread(target=work, args=m) for m in made]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for m in made:
        m[0].close()
    assert not wrong, wrong[:3]
