"""Heights of the tiled kernel's work items where a step is a launch per stage
(split domains, set_whole_step(False)): the shortest that make one wave of
resident CTAs, up to 32 rows.

The height changes which CTA computes a cell and nothing else, so a split
domain must agree bit for bit with the undivided one, whose whole-step launches
cut their rows by another rule: at sizes whose one wave takes 16, 24 and 32
rows (FP32C, 608 resident CTAs), one that needs several waves, and rows that
are no multiple of the 8-row chunk.
"""
import numpy as np
import pytest

from paper_2507_03366_gb300 import eulbfs
from paper_2507_03366_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2507_03366_gb300 import build
    build.build()


@pytest.mark.parametrize("precision,nx,ny,slabs", [
    (eulbfs.FP32C, 400, 400, 2), (eulbfs.FP32C, 600, 599, 2), (eulbfs.FP32C, 768, 768, 4), (eulbfs.FP32C, 897, 803, 3),
    (eulbfs.FP64, 512, 500, 2)])
def test_split_domain_equals_undivided(precision, nx, ny, slabs):
    case = wl.droplet(max(nx, ny), theta_deg=82.0, St=0.25, Tw=-0.6, axisymmetric=True,
                      hysteresis=(100.0, 39.0)).crop(nx, ny)
    whole = eulbfs.Solver([case], precision=precision)
    stages = eulbfs.Solver([case], precision=precision)
    stages.set_whole_step(False)
    split = eulbfs.Solver([], precision=precision)
    slots = split.add_split(case, slabs)
    for s in (whole, stages, split):
        s.step(6)
    want = whole.fields()
    for got in (stages.fields(), split.split_fields(slots)):
        for f in ("H", "T", "Fl", "C", "p", "u", "v"):
            assert np.array_equal(got[f], want[f]), f
