"""crash_kernel_time covers the whole emission of a step in bundles: in a row of
four cells, where walks are a few crossings long, most of a step is drawing and
sorting directions, and the timed transport is most of the step."""
import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native
from _common import small_hhe_box

pytestmark = pytest.mark.gpu


def test_timed_transport_of_bundles_holds_the_sort():
    torch = pytest.importorskip("torch")
    box = small_hhe_box((4, 1, 1), n_src=1, seed=790, thin=True)
    P, dt = 40_000_000, 0.01 * inputs.MYR_S
    g = native.Grid(box, native.CRASH_MIXED)
    g.set_options(chemistry=0, timing=1)
    stream = torch.cuda.ExternalStream(g.stream())
    g.step(dt, P)
    g.sync()
    shares = []
    for _ in range(5):
        g.reset_kernel_time()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        g.step(dt, P)
        e1.record(stream)
        g.sync()
        ms, n = g.kernel_time()
        assert n == 1
        shares.append(ms / e0.elapsed_time(e1))
    # the rest: preparation, budget and end of the step, some 20 us of several ms
    assert 0.9 < np.median(shares) <= 1.0
    g.close()
