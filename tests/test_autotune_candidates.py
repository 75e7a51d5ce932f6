"""The autotuner's candidates differ in what the kernels run."""
from paper_1712_09494_gb300 import autotune as at


def test_bucket_candidates_differ_in_more_than_the_lane_count():
    """lanes_per_key is accepted and checked, and no kernel depends on it."""
    cands = at.CANDIDATES["bucket"]
    kernels = [tuple(sorted((k, v) for k, v in c.items() if k != "lanes_per_key")) for c in cands]
    assert len(set(kernels)) == len(cands) == 6
    assert {c["bucket_slots"] for c in cands} == {8, 16, 32}
    # Pairs that ht_create accepts: 1 to 8 slots a lane.
    assert all(1 <= c["bucket_slots"] // c["lanes_per_key"] <= 8 for c in cands)
