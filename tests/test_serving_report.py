"""Times of a served case: its wait and its time to solution count from one
moment, its arrival, or its admission where a closed loop admits it earlier."""
from paper_2507_03366_gb300.serving import Outcome, ServeReport


def _report(*times):
    return ServeReport([Outcome(k, *t, cells=64, steps=4) for k, t in enumerate(times)], 1.0, 256, 1, 0)


def test_waits_count_from_the_arrival():
    s = _report((0.5, 0.75, 2.0), (1.0, 1.0, 3.0)).summary()
    assert s["mean_queue_s"] == 0.125
    assert s["p50_s"] == 1.75


def test_a_case_admitted_before_its_arrival_did_not_wait():
    r = _report((5.0, 0.25, 1.0), (0.0, 0.5, 1.5))
    assert [o.latency_s for o in r.outcomes] == [0.75, 1.5]
    assert r.summary()["mean_queue_s"] == 0.25
