"""Heights of work items: eulbfs_set_tile names one and the batch runs in items
of that height, 0 leaves it to the batch's size, and the autotuner keeps the
better of the two."""
import numpy as np
import pytest

from paper_2507_03366_gb300 import eulbfs
from paper_2507_03366_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CANDIDATES = (32, 48, 64, 96, 128, 160, 192, 256)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2507_03366_gb300 import build
    build.build()


def _items(cases, rows):
    """Strips x runs of round(ny / rows), in whole 8-row chunks."""
    n = 0
    for c in cases:
        chunks, per = -(-c.ny // 8), rows // 8
        n += -(-c.nx // 31) * min(chunks, max(1, (chunks + per // 2) // per))
    return n


@pytest.mark.parametrize("precision", [eulbfs.FP32C, eulbfs.FP64])
@pytest.mark.parametrize("sides", [(40, 72), (128, 400), (512, 640)])
def test_a_named_height_is_the_height_that_runs(sides, precision):
    """Batches below and above the short-item limit, at heights below and above the batch's own."""
    cases = [wl.droplet(s, theta_deg=90.0, St=0.3) for s in sides]
    s = eulbfs.Solver(cases, precision=precision)
    own = s.work_list()
    for rows in (8, 24, 64, 256):
        s.set_tile(rows)
        w = s.work_list()
        assert (w["short_items"], w["rows"], w["items"]) == (0, rows, _items(cases, rows))
    s.set_tile(0)
    assert s.work_list() == own
    assert own["short_items"] == (sides[0] < 128)


def test_autotune_leaves_a_small_batch_to_its_size():
    """Items of 32 rows and more are several times slower there than the short
    items of the batch's size, and a height picked on one case would be carried
    into every batch the solver holds later."""
    s = eulbfs.Solver([wl.droplet(128, theta_deg=90.0, St=0.3)], precision=eulbfs.FP32C)
    own = s.work_list()
    rows, ms = s.autotune(20)
    report = s.autotune_report()
    assert rows in CANDIDATES and ms == report[rows] == min(report.values())
    assert s.work_list() == own and own["short_items"]
    large = wl.film(1024)
    s.add(large)
    fresh = eulbfs.Solver([wl.droplet(128, theta_deg=90.0, St=0.3), large], precision=eulbfs.FP32C)
    assert s.work_list() == fresh.work_list()


def test_autotune_times_the_heights_it_reports():
    """On 1024 x 1024 the candidates are plans of their own: an item of 256 rows
    is swept eight times as long as one of 32, and two CTAs' worth of them
    leave most of the chip idle."""
    s = eulbfs.Solver([wl.film(1024)], precision=eulbfs.FP32C)
    s.autotune(10)
    report = s.autotune_report()
    assert sorted(report) == list(CANDIDATES)
    assert report[256] > 2.0 * report[32]


def test_work_list_arguments():
    s = eulbfs.Solver([wl.droplet(32)], precision=eulbfs.FP32C)
    assert eulbfs.lib().eulbfs_work_list(s._h, None, None, None, None) == eulbfs.OK
    assert eulbfs.lib().eulbfs_work_list(None, None, None, None, None) == eulbfs.EINVAL


@pytest.mark.parametrize("precision", [eulbfs.FP32C, eulbfs.FP64])
@pytest.mark.parametrize("n,short", [(384, 1), (400, 1), (416, 0)])
def test_the_short_kernel_ends_where_the_tiled_one_is_faster(n, short, precision):
    """4.1, 4.3 and 4.8 items of eight rows per SM; the same fields by both kernels."""
    case = wl.droplet(n, theta_deg=82.0, St=0.25, Tw=-0.6, axisymmetric=True, hysteresis=(100.0, 39.0))
    own, tiled = (eulbfs.Solver([case], precision=precision) for _ in range(2))
    assert own.work_list()["short_items"] == short
    tiled.set_tile(16)
    for s in (own, tiled):
        s.step(18)
    for f in ("H", "T", "Fl", "C", "p", "u", "v"):
        assert np.array_equal(own.fields()[f], tiled.fields()[f]), f


def test_one_wave_of_16_rows_where_a_step_is_a_launch_per_stage():
    """448 x 448 in two slabs: 420 items of 16 rows for 608 resident CTAs, above the short kernel's limit."""
    case = wl.droplet(448, theta_deg=82.0, St=0.25, Tw=-0.6, axisymmetric=True, hysteresis=(100.0, 39.0))
    split, whole = (eulbfs.Solver([], precision=eulbfs.FP32C) for _ in range(2))
    slots = split.add_split(case, 2)
    whole.add(case)
    w = split.work_list()
    assert (w["short_items"], w["rows"], w["items"]) == (0, 16, 420)
    for s in (split, whole):
        s.step(6)
    a, b = split.split_fields(slots), whole.fields()
    for f in ("H", "T", "Fl", "C", "p", "u", "v"):
        assert np.array_equal(a[f], b[f]), f
