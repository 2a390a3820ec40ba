"""The tuner's candidates for the brick schedules differ in something the march
reads: no two of them are the same solve."""
from paper_1502_07303_gb300 import autotune


def _solve(c):
    # what the brick schedules read of a candidate
    return tuple(c.get(k, 0) for k in autotune.PARAMS if k != "bucket")


def test_no_candidate_is_timed_twice():
    for search in (autotune.QUICK, None):
        got = [_solve(c) for c in autotune.candidates(search)]
        assert len(got) == len(set(got))
