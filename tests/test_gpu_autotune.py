"""The batch autotuner's candidates: the default by size, and the schedules that it
chooses from."""
import pytest

from paper_2407_12399_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

SCHEDULE = 7
CANDIDATES = (0, 8, 6, 4)


@pytest.mark.parametrize("dims", [(12, 16), (40, 48)])
def test_the_kept_schedule_is_the_fastest_candidate(dims):
    import paper_2407_12399_gb300 as tsf
    fields, _ = S.uneven_batch(n=3, seed=4, dims=dims)
    b = tsf.Batch(fields)
    old = tsf.tsf_debug_set(SCHEDULE, 5)
    try:
        choice, ms = b.autotune()
    finally:
        kept = tsf.tsf_debug_set(SCHEDULE, old)
        b.close()
    assert kept == CANDIDATES[choice]
    assert ms[choice] == min(ms)
