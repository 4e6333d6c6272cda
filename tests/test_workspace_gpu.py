"""The packet workspace a context keeps between steps: it is rebuilt when the
sources' number of colours changes the length of a queue record."""
import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native
from _common import small_hhe_box

pytestmark = pytest.mark.gpu
FIELDS = [native.F_DEP_HI, native.F_DEP_HEI, native.F_DEP_HEII, native.F_DEP_E, native.F_BUDGET]
DT = 0.01 * inputs.MYR_S


def _step(g, P, **opts):
    g.set_options(chemistry=0, **opts)
    g.set_step_index(0)
    g.step(DT, P)
    return [g.read(f) for f in FIELDS]


@pytest.mark.parametrize("passes", [dict(seg_per_iter=8, resort_interval=1, persistent=0), dict(seg_per_iter=8), dict(tile=1)])
@pytest.mark.parametrize("order", [(1, 8), (8, 1), (5, 16), (1, 8, 1, 12)])
def test_new_sources_with_other_colours_in_passes(passes, order):
    box = small_hhe_box((18, 13, 11), n_src=2, seed=780, thin=True)
    P = 2 * 4001
    g = native.Grid(box, native.CRASH_MIXED)
    for bins in order:
        E = np.array([20.0]) if bins == 1 else np.geomspace(14.0, 150.0, bins)
        g.add_sources(box.src_pos, box.src_ndot, E, np.full((2, bins), 1.0 / bins))
        got = _step(g, P, **passes)
        for a, b in zip(_step(g, P, wavefront=0), got):
            assert np.array_equal(a, b), bins
    g.close()
