"""Absorbers and fractions outside the ordinary range.  An infinite absorber is
a perfect sink of the packets that cross it and of no others: a segment of no
length (a source on a cell's corner starts one in the cell above it for every
packet that flies the other way) absorbs nothing."""
import ctypes as C
import itertools

import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native
from _common import assert_deposits_equal, pair, small_hhe_box

pytestmark = pytest.mark.gpu
DEPOSITS = [native.F_DEP_HI, native.F_DEP_HEI, native.F_DEP_HEII, native.F_DEP_E, native.F_BUDGET]
DT = 0.01 * inputs.MYR_S


def _bins(n):
    return np.array([20.0]) if n == 1 else np.geomspace(14.0, 150.0, n)


@pytest.mark.parametrize("bins,packets", list(itertools.product((1, 5, 8), (4000, 200000))))
def test_segment_of_no_length_in_an_infinite_absorber(bins, packets):
    """The sink's deposits equal those of an absorber of a finite density that
    lets nothing through (optical depths above 1e9)."""
    torch = pytest.importorskip("torch")
    box = small_hhe_box((8, 8, 8), n_src=1, seed=810)
    arrays = [np.ascontiguousarray(a, np.float64).reshape(-1) for a in
              (np.array([4.0, 4.0, 4.0]), box.src_ndot, _bins(bins), np.full(bins, 1.0 / bins))]
    pos, ndot, E, f = (a.ctypes.data_as(C.POINTER(C.c_double)) for a in arrays)
    sink = 4 + 8 * (4 + 8 * 4)
    got = []
    for density in (np.inf, 1e25):
        a = torch.full((512, 4), 1e-7, dtype=torch.float32, device="cuda")
        a[sink, 0] = density
        a[sink, 1:] = 0.0
        dep = torch.zeros((512, 4), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        budget = np.zeros(8, np.int64)
        desc = native.make_desc(box, native.CRASH_MIXED)
        st = native.lib().crash_transport_noalloc(C.byref(desc), 1, pos, ndot, bins, E, f, DT, 0, packets, 0, a.data_ptr(),
                                                  dep.data_ptr(), budget.ctypes.data_as(C.POINTER(C.c_int64)), None)
        assert st == native.CRASH_OK
        dep = dep.cpu().numpy()
        # (an infinite optical depth has no heating share; the photons and every other cell are the same)
        dep[sink, 3] = 0
        got.append((dep, budget[:5].copy()))
    (d0, b0), (d1, b1) = got
    assert np.array_equal(b0, b1) and b0[0] == b0[1] + b0[2] and b0[2] > 0.8 * b0[0]
    assert np.array_equal(d0, d1) and d0[sink, 0] > 0.1 * b0[0]


@pytest.mark.parametrize("field,value", [(native.F_XHEII, 4.5), (native.F_XHII, 1.5)])
def test_negative_absorbers_do_not_depend_on_the_order(field, value):
    """Fractions above 1 make absorbers negative; the deposits are the same in
    emission order, in bundles, in passes and in tiles."""
    box = small_hhe_box((20, 20, 20), n_src=2, seed=811)
    P = 2 * 70001
    rng = np.random.default_rng(1)
    sel = rng.choice(8000, 300, replace=False)
    out = []
    for opts in (dict(wavefront=0), dict(), dict(seg_per_iter=8), dict(tile=1)):
        g = native.Grid(box, native.CRASH_MIXED)
        g.set_options(chemistry=0, **opts)
        x = g.read(field)
        x.reshape(-1)[sel] = value
        g.write(field, x)
        g.step(DT, P)
        out.append([g.read(k) for k in DEPOSITS])
        g.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)


def test_fp64_thick_cells_with_fractions_above_one():
    """FP64 form: cells with x_HII = 1.5 dense enough that e^-tau overflows are
    transparent (the transmitted photons are clamped to those that entered):
    they absorb nothing and the photon budget closes."""
    box = small_hhe_box((12, 12, 12), n_src=2, seed=812)
    sel = np.random.default_rng(2).choice(1728, 80, replace=False)
    box.nH = box.nH.copy()
    box.nH.reshape(-1)[sel] = 1e6
    g = native.Grid(box, native.CRASH_FP64_PLAIN)
    g.set_options(chemistry=0)
    x = g.read(native.F_XHII)
    x.reshape(-1)[sel] = 1.5
    g.write(native.F_XHII, x)
    for f, v in ((native.F_XHEII, 0.0), (native.F_XHEIII, 1.0)):      # no He absorbers there either
        y = g.read(f)
        y.reshape(-1)[sel] = v
        g.write(f, y)
    g.step(DT, 2 * 6000)
    b = g.read(native.F_BUDGET)
    assert b[0] == b[1] + b[2] and 0 < b[1] <= b[0]
    for f in DEPOSITS[:4]:
        d = g.read(f).reshape(-1)
        assert (d >= 0).all() and (d[sel] == 0).all()
    g.close()


def test_fp64_he_absorbers_that_are_not_numbers():
    """FP64 form: a cell whose He absorbers are NaN takes every photon that
    enters it, of the colours below the He thresholds too, as a cell of
    infinite H I does."""
    box = small_hhe_box((12, 12, 12), n_src=2, seed=813, thin=True)
    sel = np.random.default_rng(3).choice(1728, 80, replace=False)
    out = []
    for field, value in ((native.F_XHEII, np.nan), (native.F_XHII, -np.inf)):
        g = native.Grid(box, native.CRASH_FP64_PLAIN)
        g.set_options(chemistry=0)
        x = g.read(field)
        x.reshape(-1)[sel] = value
        g.write(field, x)
        g.step(DT, 2 * 6000)
        b = g.read(native.F_BUDGET)
        assert b[0] == b[1] + b[2] and b[1] > 0 and b[2] > 0
        dep = [g.read(f).reshape(-1) for f in DEPOSITS[:4]]
        for d in dep:
            d[sel] = 0
        out.append(dep + [b[:5]])
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("bins", [1, 5, 8])
def test_crossings_of_packets_without_photons(bins):
    """A source of no luminosity on a cell's corner: its packets cross one cell,
    after up to three segments of no length, whatever the pass length."""
    box = small_hhe_box((17, 12, 16), n_src=2, seed=814, thin=True)
    box.src_pos = np.array([[11.0, 3.0, 7.0], [6.5, 0.2, 15.1]])
    box.src_ndot = np.array([0.0, 1e48])
    box.bin_eV, box.bin_frac = _bins(bins), np.full((2, bins), 1.0 / bins)
    P = 2 * 60_000
    budgets = []
    for opts in (dict(wavefront=0), dict(), dict(seg_per_iter=1), dict(seg_per_iter=2, persistent=0), dict(seg_per_iter=3),
                 dict(seg_per_iter=64), dict(tile=1)):
        g = native.Grid(box, native.CRASH_MIXED)
        g.set_options(chemistry=0, **opts)
        g.step(DT, P)
        budgets.append(g.read(native.F_BUDGET)[:5].tolist())
        g.close()
    assert all(b == budgets[0] for b in budgets), budgets
    g = native.Grid(box, native.CRASH_FP64_PLAIN)
    g.set_options(chemistry=0)
    g.step(DT, P)
    assert g.read(native.F_BUDGET)[3] == budgets[0][3]
    g.close()


@pytest.mark.parametrize("he,fractions", [(0.08, (1.0, 0.0, 1.0)), (0.08, (1.0, 0.0, 0.9)), (0.0, (1.0, 0.0, 0.0))])
def test_fp64_cells_without_absorbers(he, fractions):
    """FP64 form, cells with nothing left to absorb in some or all colours: what
    rounding N to FP64 takes off goes to H I, and no deposit is out of range;
    with He in the context (a pure-H box beside a box with He too), against the
    oracle."""
    boxes = [small_hhe_box((9, 8, 7), n_src=2, seed=815), small_hhe_box((6, 6, 6), n_src=1, seed=816)]
    boxes[0].he_over_h = he
    boxes[0].x_HII0, boxes[0].x_HeII0, boxes[0].x_HeIII0 = fractions
    boxes[0].src_ndot = np.array([1.76e42, 5.2e42])
    g = native.Grid(boxes, native.CRASH_FP64_PLAIN)
    g.set_options(chemistry=0)
    g.step(DT, [2 * 60, 700])
    for i, box in enumerate(boxes):
        _, o = pair(box)
        o.set_options(chemistry=0)
        o.step(DT, [2 * 60, 700][i])
        assert_deposits_equal(g, o, i)
        b = g.read(native.F_BUDGET, i)
        assert b[0] == b[1] + b[2]
        for f in DEPOSITS[:3]:
            assert 0 <= g.read(f, i).min() and g.read(f, i).max() <= b[1]
    g.close()
