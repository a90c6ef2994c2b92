"""D1 stages after a failed one.  On the whole-GPU rounds' path (forced here on
small fields) no kernel may use records that nobody initialised when an earlier
one failed (a union-find item that hits its step cap).  A column pool that runs
out anywhere in the D1 stages ends them in step, is doubled, and D1 starts
again."""
import pytest

import oracle

from .test_gpu_parity import NAMED, gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu

_rows = {}

ROUND_CAP, GRID_MIN, HANDOFF, PHASE_A, ROUNDS, POOL = 3, 5, 6, 7, 11, 14


def _want(name):
    if name not in _rows:
        f = NAMED[name]()
        _rows[name] = oracle_rows(f, oracle.diagram(f)["pairs"])
    return _rows[name]


class _Knobs:
    def __init__(self, knobs):
        self.knobs = knobs

    def __enter__(self):
        import paper_2407_12399_gb300 as tsf
        self.old = {k: tsf.tsf_debug_set(k, v) for k, v in self.knobs.items()}

    def __exit__(self, *exc):
        import paper_2407_12399_gb300 as tsf
        for k, v in self.old.items():
            tsf.tsf_debug_set(k, v)


@pytest.mark.parametrize("name", ["plain_32", "filament_64"])
def test_a_failed_union_find_ends_the_first_diagram_and_the_next_is_right(name):
    import paper_2407_12399_gb300 as tsf
    f = NAMED[name]()
    fld = gpu_field(f)  # its buffers are new: nothing ran before on them
    with _Knobs({GRID_MIN: 0, HANDOFF: 0, ROUND_CAP: 1}):
        r, _ = tsf.tsf_compute_diagram(fld._h, None, 0)
    assert r == tsf.TSF_ETIMEOUT, tsf.tsf_status_string(r)
    with _Knobs({GRID_MIN: 0, HANDOFF: 0}):
        got = gpu_rows(fld.diagram())
    assert got == _want(name)


# Words of the pool per critical triangle.  A column has 64 of its own from the
# start, and 84 % (plain_32) and 51 % (filament_64) of the triangles are columns:
# 4 words fail for most columns, 30 and 50 for some, 33 and 54 leave little room
# for the entries that move to the second phase (all columns with one round), for
# outputs that grow there and for the reduction's copies.
@pytest.mark.parametrize("words", [4, 30, 33, 50, 54, 60])
@pytest.mark.parametrize("knobs", [{}, {GRID_MIN: 0, HANDOFF: 0}, {GRID_MIN: 0, HANDOFF: 32, ROUNDS: 1},
                                   {ROUNDS: 1, PHASE_A: 4}], ids=str)
@pytest.mark.parametrize("name", ["plain_32", "filament_64"])
def test_a_column_pool_that_runs_out_is_doubled(name, knobs, words):
    f = NAMED[name]()
    with _Knobs({POOL: words, **knobs}):
        fld = gpu_field(f)
        got = gpu_rows(fld.diagram())
    assert got == _want(name)
