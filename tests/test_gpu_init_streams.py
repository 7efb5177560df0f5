"""A handle made on a stream of its own while the default stream is busy: what its
reductions rely on (the count of finished blocks) is in place before the first call, not
behind the default stream's work.
"""
import numpy as np
import pytest
import torch

from paper_2103_01597_gb300 import ac, build, synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    ac.load_library()
    torch.cuda.init()


@pytest.mark.parametrize("kind", ["handle", "ensemble"])
def test_first_reduction_beside_a_busy_default_stream(kind):
    n = (36, 17, 9)
    f = synthetic.smooth_state(n, 5, amp=0.3)
    want = float(np.max(f[0]))
    side = torch.cuda.Stream()
    # memory that the allocations below may be given again, all bits set
    for _ in range(4):
        junk = [torch.full((1 << 20,), 0xff, dtype=torch.uint8, device="cuda") for _ in range(8)]
        torch.cuda.synchronize()
        del junk
        torch.cuda.empty_cache()
        torch.cuda._sleep(200_000_000)  # a tenth of a second on the default stream
        with torch.cuda.stream(side):
            if kind == "handle":
                sim = ac.Simulation(n)
                sim.load(f)
                assert [sim.reduce(ac.AC_MAX, 0) for _ in range(2)] == [want, want]
            else:
                sim = ac.Batch([(n, (1.0, 1.0, 1.0), 1e-3, 1e-3)], precision=ac.AC_FP32)
                sim.load(0, f)
                assert ac.ac_batch_reduce(sim.b, 0, ac.AC_MAX, 0) == float(np.float32(want))
            sim.close()
        torch.cuda.synchronize()
