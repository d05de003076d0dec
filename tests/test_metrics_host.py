"""The benchmark's derived figures, on hand-made inputs (no GPU)."""
import numpy as np
import pytest

import bench
from paper_2509_24815_gb300 import STATS, metrics


def _stats(spans):
    st = np.zeros((len(spans), len(STATS)), dtype=np.uint64)
    st[:, STATS.index("t_start_ns")] = [a for a, _ in spans]
    st[:, STATS.index("t_end_ns")] = [b for _, b in spans]
    return st


# three slots: the fourth and fifth query start as the first two end, the last overlaps nothing
def test_resident_queries_and_occupancy():
    st = _stats([(1000, 3000), (1000, 4000), (1100, 9000), (3000, 8000), (4000, 5000), (9000, 9500)])
    assert metrics.resident_queries(st) == 3
    occ = metrics.queue_occupancy(st, 3)
    assert occ["busy"] == pytest.approx((2000 + 3000 + 7900 + 5000 + 1000 + 500) / (3 * 8500))
    assert metrics.resident_queries(_stats([(5, 6)])) == 1


# a traffic ratio holds for the workload, group and prefetch setting it was captured with
def test_traffic_ratio_needs_a_capture_of_the_form(monkeypatch):
    monkeypatch.setattr(bench, "TRAFFIC_PER_EXEC_BYTE", {("c2", 1, True): 0.5})
    form = dict(shape=1, group=1, cta_warps=0, wave=8, persistent=True, no_prefetch=False)
    assert bench.traffic_ratio("c2", form) == 0.5
    assert bench.traffic_ratio("c2", dict(form, shape=0, group=0)) == 0.5
    for other in (dict(group=8), dict(no_prefetch=True), dict(shape=2, group=8)):
        assert bench.traffic_ratio("c2", dict(form, **other)) is None
    assert bench.traffic_ratio("c3", form) is None
