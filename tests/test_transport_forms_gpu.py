"""The forms of the mixed transport give the same bits: packets in emission
order, sorted into bundles by source and direction, or in passes, at the
sizes where the forms' rules and remainders lie (one thread's worth above the
resident packets, partial warps and chunks, one source or many, each number
of colours and each set of deposited values, periodic walks, batches); the
FP64 form's bundles equal the oracle."""
import ctypes as C

import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native
from _common import assert_deposits_equal, pair, small_hhe_box

pytestmark = pytest.mark.gpu
FIELDS = [native.F_DEP_HI, native.F_DEP_HEI, native.F_DEP_HEII, native.F_DEP_E, native.F_BUDGET]
DT = 0.01 * inputs.MYR_S
RESIDENT = 152 * 3 * 256


def _deposits(boxes, P, **opts):
    g = native.Grid(boxes, native.CRASH_MIXED)
    g.set_options(chemistry=0, **opts)
    for _ in range(2):
        g.step(DT, P)
    n = len(boxes) if isinstance(boxes, list) else 1
    out = [g.read(f, b) for b in range(n) for f in FIELDS]
    g.close()
    return out


def _same(a, b, what):
    for x, y in zip(a, b):
        assert np.array_equal(x, y), what


@pytest.mark.parametrize("dims,n_src,per_src,bins,he,iso,thin,opts", [
    ((17, 12, 9), 1, RESIDENT + 1, 8, 0.08, 0, False, {}),
    ((17, 12, 9), 7, 30011, 8, 0.08, 0, True, dict(pkt_begin=3, pkt_end=29000)),
    ((33, 8, 21), 3, 60013, 8, 0.08, 0, False, dict(chunk_packets=50021)),
    ((16, 16, 16), 500, 301, 1, 0.0, 1, True, dict(chunk_packets=131)),
    ((24, 24, 24), 2, 90001, 1, 0.0, 1, False, {}),
    ((20, 20, 20), 2, 70001, 1, 0.0, 0, True, {}),
    ((20, 20, 20), 2, 70001, 8, 0.0, 0, False, {}),
    ((20, 20, 20), 2, 70001, 8, 0.08, 1, False, {}),
    ((23, 19, 13), 5, 40009, 5, 0.08, 0, False, {}),
    ((40, 1, 1), 1, 150000, 12, 0.08, 0, True, {}),
])
def test_bundles_and_passes_equal_emission_order(dims, n_src, per_src, bins, he, iso, thin, opts):
    box = small_hhe_box(dims, n_src=n_src, seed=700 + n_src, nbins=1 if bins == 1 else 8, thin=thin)
    if bins not in (1, 8):
        E, f = inputs.blackbody_bins(1e5, np.geomspace(13.6, 200.0, bins + 1))
        box.bin_eV, box.bin_frac = E, np.tile(f, (n_src, 1))
    box.he_over_h, box.isothermal = he, iso
    P = n_src * per_src
    ref = _deposits(box, P, wavefront=0, **{k: v for k, v in opts.items() if k != "chunk_packets"})
    assert ref[-1][0] == ref[-1][1] + ref[-1][2] and ref[-1][1] > 0
    # (chunks of 131 packets and 32 sources each would be thousands of launches)
    small = opts.get("chunk_packets", 1 << 20) < 1000
    if not small:
        _same(ref, _deposits(box, P, **opts), "bundles")
    else:
        _same(ref, _deposits(box, P), "bundles")
        _same(ref, _deposits(box, P, chunk_packets=131 * 301), "bundles of 131 sources")
    wide = {k: v for k, v in opts.items() if k != "chunk_packets"}
    _same(ref, _deposits(box, P, seg_per_iter=64, resort_interval=1, persistent=0, reg_cap=1, **wide), "passes")


def test_periodic_bundles_equal_emission_order():
    box = small_hhe_box((18, 11, 15), n_src=3, seed=720, thin=True)
    box.periodic = 1
    P = 3 * 45001
    _same(_deposits(box, P, wavefront=0), _deposits(box, P), "periodic")


def test_batched_bundles_equal_emission_order():
    """Bundles whose chunks start and end inside boxes, one box with an empty window."""
    boxes = [small_hhe_box((14 + 4 * i, 14, 10), n_src=1 + i, seed=730 + i) for i in range(4)]
    P = [20011, 2 * 30, 3 * 30011, 4 * 20011]
    win = dict(pkt_begin=40, pkt_end=29999)          # the second box's 30 packets a source lie outside
    ref = _deposits(boxes, P, wavefront=0, **win)
    _same(ref, _deposits(boxes, P, **win), "batch")
    _same(ref, _deposits(boxes, P, chunk_packets=33333, **win), "batch in chunks")


def test_large_grid_passes_equal_emission_order():
    """The grid and sources for which the library itself takes passes: state
    beyond L2, many sources with few packets each, buckets well filled."""
    n, n_src = 160, 4000
    rng = np.random.default_rng(5)
    E, f = inputs.blackbody_bins(1e5)
    box = inputs.Box(n=n, box_cm=6.6 * inputs.KPC_CM * n / 128, nH=None, nH0=1e-3, he_over_h=0.08, x_HII0=1 - 1e-4,
                     x_HeII0=1e-4, x_HeIII0=1 - 2e-4, T0=1e4, isothermal=0, caseB=1, z_compton=9.0, seed=741,
                     src_pos=rng.uniform(0, n, (n_src, 3)), src_ndot=rng.uniform(1e47, 1e49, n_src), bin_eV=E,
                     bin_frac=np.tile(f, (n_src, 1)))
    P = n_src * 300
    g = native.Grid(box, native.CRASH_MIXED)
    g.set_options(chemistry=0)
    before = g.launch_count()
    g.step(DT, P)
    assert g.launch_count() - before > 20            # a launch per pass
    got = [g.read(f_) for f_ in FIELDS]
    g.close()
    h = native.Grid(box, native.CRASH_MIXED)
    h.set_options(chemistry=0, wavefront=0)
    h.step(DT, P)
    _same([h.read(f_) for f_ in FIELDS], got, "passes")
    h.close()


@pytest.mark.parametrize("dims,n_src,per_src,crossings", [
    ((512, 256, 256), 100, 85000, 64),               # 2^25 cells
    ((512, 256, 257), 100, 85000, 48),
    ((512, 512, 257), 150, 113000, 32),
])
def test_pass_length_by_grid_size(dims, n_src, per_src, crossings):
    """Larger boxes take shorter passes by default; the bits are those of
    emission order."""
    rng = np.random.default_rng(6)
    E, f = inputs.blackbody_bins(1e5)
    box = inputs.Box(n=512, box_cm=6.6 * inputs.KPC_CM * 4, nH=None, nH0=1e-3, he_over_h=0.08, x_HII0=1.2e-3,
                     x_HeII0=0.0, x_HeIII0=0.0, T0=1e4, isothermal=0, caseB=1, z_compton=9.0, seed=743,
                     src_pos=rng.uniform(0, 1, (n_src, 3)) * np.array(dims), src_ndot=rng.uniform(1e47, 1e49, n_src),
                     bin_eV=E, bin_frac=np.tile(f, (n_src, 1)), dims=dims)
    out = []
    for opts in ({}, dict(wavefront=0)):
        g = native.Grid(box, native.CRASH_MIXED)
        g.set_options(chemistry=0, **opts)
        before = g.launch_count()
        g.step(DT, n_src * per_src)
        launches = g.launch_count() - before
        out.append([g.read(f_) for f_ in (native.F_DEP_HI, native.F_DEP_E, native.F_BUDGET)])
        g.close()
        if not opts:       # every pass but the last sorts (four launches); the walk crosses at most the three edges
            passes = -(-(sum(dims) + 3) // crossings) + 1
            assert 5 * passes - 4 <= launches <= 5 * passes + 8
    _same(*out, "passes")


@pytest.mark.parametrize("per_src", [7, 30000, 260000])
def test_noalloc_bundles_equal_emission_order(per_src):
    """The allocation-free call: all at once, one bundle chunk, several."""
    torch = pytest.importorskip("torch")
    box = small_hhe_box((21, 18, 13), n_src=5, seed=750)
    P = 5 * per_src
    h = native.Grid(box, native.CRASH_MIXED)
    h.set_options(chemistry=0, wavefront=0)
    h.step(DT, P)
    nH = torch.from_numpy(np.ascontiguousarray(box.nH, np.float32).reshape(-1)).cuda().double()
    a = torch.zeros((nH.numel(), 4), dtype=torch.float64, device="cuda")
    nHe = nH * box.he_over_h
    a[:, 0], a[:, 1], a[:, 2] = nH * (1.0 - box.x_HII0), nHe * ((1.0 - box.x_HeII0) - box.x_HeIII0), nHe * box.x_HeII0
    a = a.float()
    dep = torch.zeros((nH.numel(), 4), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    arrays = [np.ascontiguousarray(x, np.float64).reshape(-1) for x in (box.src_pos, box.src_ndot, box.bin_eV, box.bin_frac)]
    pos, ndot, E, f = (x.ctypes.data_as(C.POINTER(C.c_double)) for x in arrays)
    budget = np.zeros(8, np.int64)
    desc = native.make_desc(box, native.CRASH_MIXED)
    st = native.lib().crash_transport_noalloc(C.byref(desc), 5, pos, ndot, len(arrays[2]), E, f, DT, 0, P, 0, a.data_ptr(),
                                              dep.data_ptr(), budget.ctypes.data_as(C.POINTER(C.c_int64)), None)
    assert st == native.CRASH_OK
    got = dep.cpu().numpy()
    for k, f_ in enumerate(FIELDS[:4]):
        assert np.array_equal(h.read(f_).reshape(-1), got[:, k]), f_
    assert np.array_equal(h.read(native.F_BUDGET)[:5], budget[:5])
    h.close()


@pytest.mark.parametrize("dims,n_src,per_src,bins,he,thin,opts", [
    ((14, 11, 9), 1, 8191, 8, 0.08, False, {}),          # below the bundles' rule, and at it
    ((14, 11, 9), 1, 8192, 8, 0.08, False, {}),
    ((14, 11, 9), 3, 4001, 8, 0.08, True, dict(chunk_packets=3001)),
    ((12, 12, 12), 2, 5003, 1, 0.0, False, {}),
    ((12, 9, 7), 2, 4500, 5, 0.08, False, dict(pkt_begin=17)),
])
def test_fp64_bundles_equal_the_oracle(dims, n_src, per_src, bins, he, thin, opts):
    box = small_hhe_box(dims, n_src=n_src, seed=760 + n_src, nbins=1 if bins == 1 else 8, thin=thin)
    if bins not in (1, 8):
        E, f = inputs.blackbody_bins(1e5, np.geomspace(13.6, 200.0, bins + 1))
        box.bin_eV, box.bin_frac = E, np.tile(f, (n_src, 1))
    box.he_over_h = he
    g, o = pair(box)
    g.set_options(chemistry=0, **opts)
    o.set_options(chemistry=0, **{k: v for k, v in opts.items() if k != "chunk_packets"})
    for _ in range(2):
        g.step(DT, n_src * per_src)
        o.step(DT, n_src * per_src)
        assert_deposits_equal(g, o)
    g.close()


def test_fp64_step_without_room_to_sort_runs(monkeypatch):
    box = small_hhe_box((10, 10, 10), n_src=1, seed=770)
    monkeypatch.setenv("CRASH_DEVICE_MEMORY_CAP", str(250000))     # the grid's 150 kB, not 20000 packets' sort
    g, o = pair(box)
    g.step(DT, 20000)
    o.step(DT, 20000)
    assert_deposits_equal(g, o)
    g.close()
