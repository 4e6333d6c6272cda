"""Which form the library takes by itself, by the kernels a step launches, and
that its deposits are those of emission order: passes (many launches) for
sources of few packets in any grid once there are packets enough to sort,
bundles for sources of many packets, one field or a batch."""
import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native

pytestmark = pytest.mark.gpu
DT = 0.01 * inputs.MYR_S
FIELDS = [native.F_DEP_HI, native.F_DEP_E, native.F_BUDGET]


def _box(n, n_src, seed):
    rng = np.random.default_rng(seed)
    E, f = inputs.blackbody_bins(1e5)
    return inputs.Box(n=n, box_cm=6.6 * inputs.KPC_CM * n / 128, nH=None, nH0=1e-3, he_over_h=0.08, x_HII0=1 - 1e-4,
                      x_HeII0=1e-4, x_HeIII0=1 - 2e-4, T0=1e4, isothermal=0, caseB=1, z_compton=9.0, seed=seed,
                      src_pos=rng.uniform(0, n, (n_src, 3)), src_ndot=rng.uniform(1e47, 1e49, n_src), bin_eV=E,
                      bin_frac=np.tile(f, (n_src, 1)))


SEVERAL = (32, 48, 64, 96, 128)


@pytest.mark.parametrize("n,boxes,n_src,per_src,passes", [
    (256, 1, 100_000, 40, True),         # few packets per source, fewer than a quarter of the cells in all
    (128, 1, 100_000, 10, True),         # the same in a grid that fits L2
    (64, 8, 1000, 100, True),            # and in a batch
    (64, 8, 1000, 65, False),            # under 2^19 packets
    (256, 1, 100, 6_000, True),          # w = 33 cells, 26 at 0.036 packets per cell
    (256, 1, 30, 30_000, False),         # 15, 22 at 0.054
    (128, 1, 10, 60_000, False),
    (64, 8, 5, 20_000, False),
    (SEVERAL, 5, 30, 16_000, False),     # bundles 7 cells wide in the mean
    (SEVERAL, 5, 3000, 400, True),       # 45
    (SEVERAL, 5, 300, 800, False),       # 32, but few packets for the passes the largest box needs
])
def test_form_by_sizes(n, boxes, n_src, per_src, passes):
    batch = [_box(n if isinstance(n, int) else n[b], n_src, 820 + b) for b in range(boxes)]
    out = []
    for opts in ({}, dict(wavefront=0)):
        g = native.Grid(batch, native.CRASH_MIXED)
        g.set_options(chemistry=0, **opts)
        before = g.launch_count()
        g.step(DT, [n_src * per_src] * boxes)
        launches = g.launch_count() - before
        out.append([g.read(f, b) for b in range(boxes) for f in FIELDS])
        g.close()
        if not opts:
            # budget, preparation and end of the step, and the sort and trace of one chunk
            assert launches == 3 + 4 if not passes else launches > 20
    for a, b in zip(*out):
        assert np.array_equal(a, b)
