"""The packet workspace a context keeps between steps: it is rebuilt when the
sources' number of colours changes the length of a queue record; a step
without room for it beside an earlier step's takes its place, and one without
room for it alone runs in a form that needs less, unless passes were asked
for; a step in emission order that was asked for gives it back."""
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


def test_passes_after_bundles_where_either_has_room(monkeypatch):
    box = small_hhe_box((20, 20, 20), n_src=1, seed=781, thin=True)
    ref, g = native.Grid(box, native.CRASH_MIXED), native.Grid(box, native.CRASH_MIXED)
    # 0.7 MB of grid; the sort of 10^6 packets takes 16 MB, the queue of 10^5 14 MB
    monkeypatch.setenv("CRASH_DEVICE_MEMORY_CAP", str(20_000_000))
    for P, opts in [(1_000_000, {}), (100_000, dict(seg_per_iter=8)), (1_000_000, {}), (100_000, dict(seg_per_iter=8))]:
        want = _step(ref, P, wavefront=0)
        before = g.launch_count()
        for a, b in zip(want, _step(g, P, **opts)):
            assert np.array_equal(a, b), P
        launches = g.launch_count() - before
        assert launches == 7 if not opts else launches >= 4
    g.close()
    ref.close()


@pytest.mark.parametrize("cap,launches", [(42_000_000, 3 + 4), (30_000_000, 3 + 1)])
def test_passes_of_the_library_without_room(monkeypatch, cap, launches):
    """Sources of few packets, for which the library takes passes (140 MB of
    queue beside 22 MB of grid): bundles (16 MB) under one cap, emission order
    under the other; passes asked for are refused, and nothing is lost by it."""
    box = small_hhe_box((64, 64, 64), n_src=10_000, seed=782, thin=True)
    P = 10_000 * 100
    ref, g = native.Grid(box, native.CRASH_MIXED), native.Grid(box, native.CRASH_MIXED)
    want = _step(ref, P, wavefront=0)
    before = ref.launch_count()
    _step(ref, P)
    assert ref.launch_count() - before > 20          # (passes, where there is room)
    monkeypatch.setenv("CRASH_DEVICE_MEMORY_CAP", str(cap))
    before = g.launch_count()
    for a, b in zip(want, _step(g, P)):
        assert np.array_equal(a, b)
    assert g.launch_count() - before == launches
    with pytest.raises(native.CrashError) as e:
        _step(g, P, seg_per_iter=32)
    assert e.value.status == native.CRASH_ERR_OOM
    for a, b in zip(want, _step(g, P)):
        assert np.array_equal(a, b)
    g.close()
    ref.close()


def test_emission_order_gives_the_workspace_back():
    torch = pytest.importorskip("torch")
    box = small_hhe_box((16, 16, 16), n_src=2, seed=783)
    g = native.Grid(box, native.CRASH_MIXED)
    _step(g, 1000, wavefront=0)
    g.sync()
    free0 = torch.cuda.mem_get_info()[0]
    _step(g, 2_000_000, seg_per_iter=64)             # a queue of 2e6 records: 280 MB
    assert torch.cuda.mem_get_info()[0] < free0 - 200_000_000
    _step(g, 1000, wavefront=0)
    assert torch.cuda.mem_get_info()[0] > free0 - 50_000_000
    g.close()
