"""D1 column reduction on warps and blocks (k_d1_columns, k_d1_long).

The default schedule reduces most columns of a small field on warps.  The
tuning knobs force the other paths on the same fields: columns that go to a
block after one addition or at once (no room on the warp), blocks that keep
one or two groups of 1024 rows in shared memory and the rest in global
memory, and blocks resuming the lists that the whole-GPU rounds leave.  The
pairs are those of the oracle's plain reduction, whatever the schedule.
"""
import pytest

import oracle

from .test_gpu_parity import NAMED, gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu

CAP, ADDS, WINDOW, GRID_MIN, HANDOFF = 9, 12, 13, 5, 6


@pytest.mark.parametrize("knobs", [{ADDS: 1}, {ADDS: 1, WINDOW: 1}, {CAP: 0, WINDOW: 1}, {CAP: 0, WINDOW: 2},
                                   {CAP: 0, GRID_MIN: 0, HANDOFF: 32, WINDOW: 1}, {ADDS: 1 << 16, CAP: 1 << 16}],
                         ids=str)
@pytest.mark.parametrize("name", ["plain_32", "filament_40", "filament_64", "ring_21"])
def test_columns_on_warps_and_blocks_match_the_oracle(name, knobs):
    import paper_2407_12399_gb300 as tsf
    f = NAMED[name]()
    old = {k: tsf.tsf_debug_set(k, v) for k, v in knobs.items()}
    try:
        got = gpu_rows(gpu_field(f).diagram())
    finally:
        for k, v in old.items():
            tsf.tsf_debug_set(k, v)
    assert got == oracle_rows(f, oracle.diagram(f)["pairs"])
