"""Stage times: D0 and D2 pairs are timed apart, in launches of their own, and
profiling changes no result."""
import pytest

from .test_gpu_parity import NAMED, gpu_field, gpu_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["plain_32", "filament_40", "linear", "constant"])
def test_d0_and_d2_pairs_are_timed_apart(name):
    import paper_2407_12399_gb300 as tsf
    f = NAMED[name]()
    plain, timed = gpu_field(f), gpu_field(f)
    tsf.tsf_profile_enable(timed._h, 1)
    launches, rows = [], []
    for fld in (plain, timed):
        before = tsf.tsf_kernel_launches()
        rows.append(gpu_rows(fld.diagram()))
        launches.append(tsf.tsf_kernel_launches() - before)
    assert rows[0] == rows[1]
    stages = tsf.tsf_profile_read(timed._h)
    ms, calls = zip(stages["pairs_d0"], stages["pairs_d2"])
    assert calls == (1, 1)
    if name in ("plain_32", "filament_40"):  # lines, union-find and kills of each
        assert launches[1] - launches[0] == 3
        assert min(ms) > 0
