"""crash_autotune times the form a full step takes: its trials trace a window of
the packet ids, but the library's own form is that of the full step, with the
library's own blocks."""
import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native

pytestmark = pytest.mark.gpu
DT = 0.01 * inputs.MYR_S


def _box(n, n_src):
    rng = np.random.default_rng(9)
    E, f = inputs.blackbody_bins(1e5)
    return inputs.Box(n=n, box_cm=6.6 * inputs.KPC_CM * n / 128, nH=None, nH0=1e-3, he_over_h=0.08, x_HII0=1 - 1e-4,
                      x_HeII0=1e-4, x_HeIII0=1 - 2e-4, T0=1e4, isothermal=0, caseB=1, z_compton=9.0, seed=9,
                      src_pos=rng.uniform(0, n, (n_src, 3)), src_ndot=rng.uniform(1e47, 1e49, n_src), bin_eV=E,
                      bin_frac=np.tile(f, (n_src, 1)))


def _launches(g, P, **opts):
    g.set_options(chemistry=0, **opts)
    before = g.launch_count()
    g.step(DT, P)
    return g.launch_count() - before


@pytest.mark.parametrize("n,n_src,per_src,bundles", [
    (64, 4, 50_000, True),            # no window: 2e5 packets
    (96, 100, 1_700_000, True),       # 1.7e8 packets in a window of 6.7e7, bundles either way
    (48, 100_000, 1100, True),        # 1100 packets of a source: bundles 14.5 cells wide; the window's 671: 18.6, passes
    (48, 100_000, 800, False),        # 17.0 and 18.6: passes either way
])
def test_trials_take_the_form_of_the_full_step(n, n_src, per_src, bundles):
    P = n_src * per_src
    g = native.Grid(_box(n, n_src), native.CRASH_MIXED)
    # launches of a trial in passes depend on its pass length and sort interval only
    grid = {(s, r): _launches(g, P, pkt_end=1, seg_per_iter=s, resort_interval=r, persistent=0)
            for s in (16, 32, 64) for r in (1, 2)}
    tile = _launches(g, P, pkt_end=1, resort_interval=1, tile=1)
    full = _launches(g, P)
    assert (full == 7) == bundles
    g.set_options(chemistry=0)
    before = g.launch_count()
    block, seg, resort, reg_cap, tiles, curve = g.autotune(DT, [P])
    spent = g.launch_count() - before
    o = g.get_options()
    # two steps a trial: twelve trials in passes of either register cap and
    # block size, tiles, the library's own form; and, for passes, the sort
    # curve and the one persistent launch
    spent -= 2 * (4 * sum(grid.values()) + tile)
    if seg:
        assert block in (128, 256)
        spent -= 2 * (grid[seg, resort] + 3 + 1)
    elif not tiles:
        assert (block, resort, reg_cap, curve) == (0, 0, 0, 0) and o["persistent"] == 1
    assert spent == 2 * full
    g.close()
