"""The D1 Morse boundaries' schedules that no small diagram takes by itself: a
quarter of a warp per column with 32 + 64 entries (8, the default from 2^19
critical triangles on), with the chains and rounds that go with it there, and one
warp with 256 + 512 (2).  Any schedule gives the oracle's pairs."""
import pytest

import oracle
from paper_2407_12399_gb300 import synthetic as S

from .test_gpu_parity import NAMED, gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu

SCHEDULE, CHAIN, ROUNDS = 7, 10, 11
FIELDS = {name: NAMED[name] for name in ("plain_32", "filament_40", "filament_64", "ring_21")}
FIELDS["noise_46"] = lambda: S.gaussian_mixture((46, 47, 48), n_bumps=8, seed=5, noise_frac=0.3)
_rows = {}


@pytest.mark.parametrize("knobs", [{SCHEDULE: 2}, {SCHEDULE: 8}, {SCHEDULE: 8, CHAIN: 1, ROUNDS: 128},
                                   {SCHEDULE: 8, CHAIN: 1, ROUNDS: 2}], ids=str)
@pytest.mark.parametrize("name", sorted(FIELDS))
def test_schedules_of_large_diagrams_match_the_oracle(name, knobs):
    import paper_2407_12399_gb300 as tsf
    f = FIELDS[name]()
    if name not in _rows:
        _rows[name] = oracle_rows(f, oracle.diagram(f)["pairs"])
    old = {k: tsf.tsf_debug_set(k, v) for k, v in knobs.items()}
    try:
        got = gpu_rows(gpu_field(f).diagram())
    finally:
        for k, v in old.items():
            tsf.tsf_debug_set(k, v)
    assert got == _rows[name]
