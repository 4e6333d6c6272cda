"""Steps replayed from a CUDA graph in every form the library takes: bundles
(whose first source, key count and direction bits are host values of the
capture), the library's passes, one persistent launch and a launch per pass,
and the FP64 form's bundles; over several steps, with the number of packets
changing in between and back, the state evolving, against plain steps.  The
forms are told by the kernels a step launches."""
import numpy as np
import pytest

from paper_1101_4127_gb300 import inputs, native
from _common import DEP_FIELDS, STATE_FIELDS, small_hhe_box

pytestmark = pytest.mark.gpu
DT = 0.01 * inputs.MYR_S


def _fields(g, boxes=1):
    return [g.read(f, b) for b in range(boxes) for f, _ in STATE_FIELDS + DEP_FIELDS] + \
           [g.read(native.F_BUDGET, b) for b in range(boxes)]


def _run(boxes, precision, steps, **opts):
    """Fields after every step, and the kernels of each step."""
    g = native.Grid(boxes, precision)
    g.set_options(**opts)
    fields, launches = [], []
    for P in steps:
        before = g.launch_count()
        g.step(DT, P)
        launches.append(g.launch_count() - before)
        fields.append(_fields(g, len(boxes) if isinstance(boxes, list) else 1))
    g.close()
    return fields, launches


def _same(a, b):
    for step, (x, y) in enumerate(zip(a, b)):
        for f, (u, v) in enumerate(zip(x, y)):
            assert np.array_equal(u, v), (step, f)


@pytest.mark.parametrize("opts,launches", [
    (dict(), lambda n: n == 4 + 4),
    (dict(chunk_packets=50_021), lambda n: n % 4 == 0 and n > 8),
    (dict(pkt_begin=7, pkt_end=100_000), lambda n: n == 4 + 4),
    (dict(seg_per_iter=16, resort_interval=1, persistent=1), lambda n: n == 4 + 1),
    (dict(seg_per_iter=16, resort_interval=2, persistent=0), lambda n: n > 8),
    (dict(tile=1), lambda n: n > 8),
])
def test_replayed_steps_equal_emission_order(opts, launches):
    box = small_hhe_box((18, 15, 11), n_src=3, seed=830)
    steps = [3 * 60_001, 3 * 60_001, 3 * 90_007, 3 * 60_001, 3 * 60_001]
    window = {k: v for k, v in opts.items() if k.startswith("pkt")}
    ref, _ = _run(box, native.CRASH_MIXED, steps, wavefront=0, **window)
    got, n = _run(box, native.CRASH_MIXED, steps, use_graph=1, **opts)
    assert all(launches(k) for k in n), n
    _same(ref, got)


def test_replayed_batch_in_bundles():
    boxes = [small_hhe_box((14 + 3 * i, 14, 10), n_src=1 + i, seed=831 + i) for i in range(3)]
    P = [50_000, 2 * 40_000, 3 * 20_000]
    steps = [P, P, [2 * p for p in P], P]
    ref, _ = _run(boxes, native.CRASH_MIXED, steps, wavefront=0)
    got, n = _run(boxes, native.CRASH_MIXED, steps, use_graph=1)
    assert n == [8] * 4
    _same(ref, got)


def test_replayed_passes_of_the_library():
    """Sources of few packets: passes for 6e5 packets, bundles for 2e5, and back."""
    box = small_hhe_box((40, 40, 40), n_src=2000, seed=835)
    steps = [600_000, 600_000, 200_000, 600_000, 600_000]
    ref, _ = _run(box, native.CRASH_MIXED, steps, wavefront=0)
    got, n = _run(box, native.CRASH_MIXED, steps, use_graph=1)
    assert n[2] == 8 and all(k > 12 for k in n[:2] + n[3:]), n
    _same(ref, got)


def test_hilbert_ordered_passes_and_periodic_bundles():
    """Options whose default form is emission order at a few thousand packets, in
    the forms they are about."""
    box = small_hhe_box((20, 14, 9), n_src=3, seed=836)
    steps = [3 * 50_001] * 2
    ref, _ = _run(box, native.CRASH_MIXED, steps, wavefront=0)
    for persistent in (0, 1):
        got, n = _run(box, native.CRASH_MIXED, steps, seg_per_iter=8, resort_interval=1, sort_curve=1, persistent=persistent)
        assert n[0] == 5 if persistent else n[0] > 8
        _same(ref, got)
    box.periodic = 1
    ref, n0 = _run(box, native.CRASH_MIXED, steps, wavefront=0)
    got, n1 = _run(box, native.CRASH_MIXED, steps, use_graph=1)
    assert n0 == [5, 5] and n1 == [8, 8]
    _same(ref, got)


def test_replayed_fp64_bundles():
    box = small_hhe_box((12, 11, 9), n_src=2, seed=837)
    steps = [2 * 6000, 2 * 6000, 2 * 2000, 2 * 6000]
    ref, _ = _run(box, native.CRASH_FP64_PLAIN, steps)
    got, n = _run(box, native.CRASH_FP64_PLAIN, steps, use_graph=1, chunk_packets=5_000)
    assert n == [4 + 3 * 4, 4 + 3 * 4, 5, 4 + 3 * 4]
    _same(ref, got)
