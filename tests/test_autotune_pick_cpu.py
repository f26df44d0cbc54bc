"""The autotuner's choice (CPU): the fastest call on device buffers, and among
those within 1% of it the fastest call on host buffers."""
from paper_1806_04374_gb300 import autotune


def _r(groups, ms, host_ms=None):
    r = {"groups": groups, "refine_blocks_per_sm": 16, "score_stages": 2, "ms": ms}
    return r if host_ms is None else dict(r, host_ms=host_ms)


def test_near_ties_go_to_the_host_call():
    results = [_r(1, 7.90, 8.00), _r(2, 7.03, 8.55), _r(3, 7.06, 8.25)]
    assert [r["groups"] for r in autotune.near_best(results)] == [2, 3]
    assert autotune.pick(results)["groups"] == 3
    # host calls within 1% of each other: the device call
    assert autotune.pick([_r(2, 7.03, 8.55), _r(4, 7.05, 8.28), _r(3, 7.06, 8.25)])["groups"] == 4
    # 1.5% behind on device buffers: not a tie
    assert autotune.pick([_r(2, 7.03, 8.55), _r(3, 7.14, 8.25)])["groups"] == 2
    # no host figures, or equal ones: the device call
    assert autotune.pick([_r(2, 7.03), _r(3, 7.06)])["groups"] == 2
    assert autotune.pick([_r(3, 7.06, 8.0), _r(2, 7.03, 8.0)])["groups"] == 2
