"""The two-CTAs-per-SM instances of the short-item kernel (FP32C with its
narrowing halo, FP64 in 8 warps) against the tiled kernel, bit for bit, on
every kind of domain: walled, hysteresis, periodic, axisymmetric and with
streaming steps, at item heights from four rows to the instances' most and with
strip and row remainders.  And the bounded wait for a neighbour's item in each
kernel."""
import time

import numpy as np
import pytest

from paper_2507_03366_gb300 import eulbfs
from paper_2507_03366_gb300 import workloads as wl
from test_gpu_short_items import FIELDS, _built, _case  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [("xy", 400, 200), ("hyst", 218, 400), ("rz", 200, 200), ("rz", 333, 251), ("gen", 256, 251),
          ("gen_rz", 187, 211), ("per_x", 250, 333), ("per_y", 333, 250), ("per_y", 1024, 90), ("hyst", 33, 1500)]


@pytest.mark.parametrize("precision", [eulbfs.FP32C, eulbfs.FP64])
@pytest.mark.parametrize("kind,nx,ny", SHAPES)
def test_two_per_sm_equals_tiled_items(kind, nx, ny, precision):
    case = _case("rz" if kind == "gen_rz" else kind, nx, ny)
    if kind == "gen_rz":
        case.dt_h, case.dt_f, case.dt_g = 0.3, 0.4, 0.3
    steps = 18                                     # more than one launch
    tiled = eulbfs.Solver([case], precision=precision)
    tiled.set_tile(24)
    assert not tiled.work_list()["short_items"]
    short = eulbfs.Solver([case], precision=precision)
    w = short.work_list()
    assert (w["short_items"], w["ctas_per_sm"]) == (1, 2)
    stages = eulbfs.Solver([case], precision=precision)
    stages.set_whole_step(False)
    assert stages.work_list() == w
    for s in (tiled, short, stages):
        s.step(steps)
    want = tiled.fields()
    for got in (short.fields(), stages.fields()):
        for f in FIELDS:
            assert np.array_equal(got[f], want[f]), f


@pytest.mark.parametrize("precision", [eulbfs.FP32C, eulbfs.FP64])
@pytest.mark.parametrize("rows", [0, 8])
def test_bounded_neighbour_wait_of_each_kernel(rows, precision):
    """With probe 2 no item marks itself done: the items of the second stage
    wait out their bound (about a second), and the host reads ETIMEOUT."""
    s = eulbfs.Solver([wl.droplet(96, theta_deg=90.0, St=0.3)], precision=precision)
    s.set_tile(rows)
    assert s.work_list()["short_items"] == (rows == 0)
    eulbfs._check(eulbfs.lib().eulbfs_set_tile_wait_probe(s._h, 2))
    t0 = time.perf_counter()
    s.step(1)
    with pytest.raises(eulbfs.EulbfsError) as e:
        s.sync()
    assert e.value.code == eulbfs.ETIMEOUT
    assert time.perf_counter() - t0 < 60.0
    s.close()
