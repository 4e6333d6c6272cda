"""Tile passes: whole warps walk together, lanes whose packet has left its tile
keeping their place until the last is done.  The deposits are those of
emission order at the sizes where lanes end apart: partial warps, ragged
tiles, packets that leave after one cell or cross a whole tile, each number
of colours and each set of deposited values."""
import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native
from _common import small_hhe_box

pytestmark = pytest.mark.gpu
FIELDS = [native.F_DEP_HI, native.F_DEP_HEI, native.F_DEP_HEII, native.F_DEP_E, native.F_BUDGET]
DT = 0.01 * inputs.MYR_S


@pytest.mark.parametrize("dims,n_src,per_src,bins,he,iso,thin", [
    ((33, 17, 16), 3, 2011, 8, 0.08, 0, True),
    ((33, 17, 16), 3, 2011, 8, 0.08, 0, False),
    ((50, 20, 20), 1, 33, 1, 0.0, 1, True),
    ((16, 16, 16), 40, 31, 5, 0.08, 0, False),
    ((47, 1, 3), 2, 5000, 8, 0.0, 0, True),
    ((31, 18, 17), 5, 999, 12, 0.08, 1, True),
])
def test_tile_passes_equal_emission_order(dims, n_src, per_src, bins, he, iso, thin):
    box = small_hhe_box(dims, n_src=n_src, seed=800 + n_src, thin=thin)
    E = np.array([20.0]) if bins == 1 else np.geomspace(14.0, 150.0, bins)
    box.bin_eV, box.bin_frac = E, np.full((n_src, bins), 1.0 / bins)
    box.he_over_h, box.isothermal = he, iso
    out = []
    for opts in (dict(wavefront=0), dict(tile=1)):
        g = native.Grid(box, native.CRASH_MIXED)
        g.set_options(chemistry=0, **opts)
        g.step(DT, n_src * per_src)
        g.step(DT, n_src * per_src)
        out.append([g.read(f) for f in FIELDS])
        g.close()
    assert out[0][-1][0] == out[0][-1][1] + out[0][-1][2] and out[0][-1][1] > 0
    for a, b in zip(*out):
        assert np.array_equal(a, b)
