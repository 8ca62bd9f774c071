"""The short-item kernel (batches with too few cells to fill the chip) against
the tiled kernel.

A small domain alone runs in short items; the same domain in a batch with a
1024 x 1024 one runs in the tiled kernel's.  Every cell's arithmetic is the
same in both, so the fields must agree bit for bit: at item heights from one
row to the kernel's eight (the domain's size sets them), at strip and row
remainders, on walled, periodic, hysteresis, axisymmetric and
general-streaming domains, in one launch for many steps, per stage, and split
into slabs.
"""
import numpy as np
import pytest

from paper_2507_03366_gb300 import eulbfs
from paper_2507_03366_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

FIELDS = ("H", "T", "Fl", "C", "p", "u", "v")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2507_03366_gb300 import build
    build.build()


@pytest.fixture(scope="module")
def big():
    return wl.film(1024)


def _case(kind, nx, ny):
    rng = np.random.default_rng(nx * 1000 + ny)
    side = max(nx, ny, 32)
    case = wl.droplet(side, theta_deg=82.0, St=0.25, Tw=-0.6, axisymmetric=kind == "rz",
                      hysteresis=(100.0, 39.0) if kind in ("rz", "hyst") else None).crop(nx, ny)
    if kind == "gen":
        case.dt_h, case.dt_f, case.dt_g = 0.3, 0.4, 0.3
    if kind == "per_y":
        case.bc = wl.BC(case.bc.ylo, wl.Side(wl.ADIABATIC, wl.OUTLET, wl.NOFLUX), wl.PER, wl.PER)
    if kind == "per_x":
        case.bc = wl.BC(wl.PER, wl.PER, case.bc.ylo, wl.Side(wl.ADIABATIC, wl.OUTLET, wl.NOFLUX))
    if kind in ("per_x", "per_y"):   # a flat interface, which the periodic axis continues
        z = np.arange(ny if kind == "per_x" else nx) + 0.5
        layer = 0.5 * (1.0 + np.tanh(2.0 * (0.5 * len(z) - z) / case.props.xi))
        layer = layer[:, None] if kind == "per_x" else layer[None, :]
        case.init["C"] = np.ascontiguousarray(np.broadcast_to(layer, (ny, nx)))
    case.init["T"] = case.init["T"] + 0.05 * rng.standard_normal((ny, nx))
    case.init["u"] = 1e-3 * rng.standard_normal((ny, nx)) * case.init["C"]
    return case


SHAPES = [("xy", 2, 2), ("hyst", 31, 7), ("rz", 32, 8), ("per_y", 33, 9), ("per_x", 63, 17), ("gen", 62, 15),
          ("rz", 94, 120), ("hyst", 157, 161), ("per_y", 256, 4), ("xy", 270, 333)]


@pytest.mark.parametrize("precision", [eulbfs.FP32C, eulbfs.FP64])
@pytest.mark.parametrize("kind,nx,ny", SHAPES)
def test_short_items_equal_tiled_items(kind, nx, ny, precision, big):
    case = _case(kind, nx, ny)
    steps = 18                                     # more than one launch
    tiled = eulbfs.Solver([case, big], precision=precision)
    tiled.step(steps)
    alone = eulbfs.Solver([case], precision=precision)
    alone.step(steps)
    stages = eulbfs.Solver([case], precision=precision)
    stages.set_whole_step(False)
    stages.use_graphs(6)
    stages.step(steps)
    want = tiled.fields(0)
    for got in (alone.fields(), stages.fields()):
        for f in FIELDS:
            assert np.array_equal(got[f], want[f]), f
    if ny >= 16:
        split = eulbfs.Solver([], precision=precision)
        slots = split.add_split(case, 2)
        split.step(steps)
        got = split.split_fields(slots)
        for f in FIELDS:
            assert np.array_equal(got[f], want[f]), f
