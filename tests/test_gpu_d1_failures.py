"""D1 stages after a failed one: on the whole-GPU rounds' path (forced here on
small fields) no kernel may use records that nobody initialised when an earlier
one failed (a union-find item that hits its step cap)."""
import pytest

import oracle

from .test_gpu_parity import NAMED, gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu

ROUND_CAP, GRID_MIN, HANDOFF = 3, 5, 6


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
    assert got == oracle_rows(f, oracle.diagram(f)["pairs"])
