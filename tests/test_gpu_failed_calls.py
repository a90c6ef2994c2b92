"""Calls that fail, and the calls after them: no diagram or assignment of earlier
values is taken for the current one.  A call that only looks leaves both."""
import numpy as np
import pytest

import oracle
from paper_2407_12399_gb300 import synthetic as S

from .test_gpu_parity import NAMED, bits, gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu

ROUND_CAP = 3


def test_nothing_of_earlier_values_is_returned_for_a_nan_field():
    import paper_2407_12399_gb300 as tsf
    f = NAMED["plain_32"]()
    fld = gpu_field(f)
    fld.set_threshold(0.1)
    bad = f.copy()
    bad[3, 4, 5] = np.nan
    for call in (lambda: fld.loss_and_grad(bad), fld.diagram, lambda: fld.step(stop_s=0.0), fld.simplify):
        with pytest.raises(tsf.TsfError) as e:
            call()
        assert e.value.code == tsf.TSF_ENAN
    rng = np.random.default_rng(5)
    g = (f + rng.uniform(-0.01, 0.01, f.shape)).astype(np.float32)
    loss, grad = fld.loss_and_grad(g)
    other = gpu_field(f)
    other.set_threshold(0.1)
    want_loss, want = other.loss_and_grad(g)
    assert loss == want_loss and np.array_equal(grad.view(np.uint64), want.view(np.uint64))
    assert gpu_rows(fld.diagram()) == oracle_rows(g, oracle.diagram(g)["pairs"])


@pytest.mark.parametrize("name,tau", [("plain_32", 0.1), ("filament_64", 0.05)])
def test_a_step_after_a_failed_one_matches_the_current_diagram(name, tau):
    """The failed step has moved the values; the next one starts from their
    diagram, matched as without the reuse of the previous assignment."""
    import paper_2407_12399_gb300 as tsf
    f = NAMED[name]()
    fld = gpu_field(f)
    fld.set_threshold(tau)
    old = tsf.tsf_debug_set(ROUND_CAP, 1)
    try:
        with pytest.raises(tsf.TsfError) as e:
            fld.step(stop_s=0.0)
    finally:
        tsf.tsf_debug_set(ROUND_CAP, old)
    assert e.value.code == tsf.TSF_ETIMEOUT
    want = gpu_field(f)
    want.set_threshold(tau)
    want.step(stop_s=0.0, fast_assignment_update=0)
    assert np.array_equal(bits(fld.values()), bits(want.values()))
    assert gpu_rows(fld.diagram()) == gpu_rows(want.diagram())
    for _ in range(2):
        fld.step(stop_s=0.0)
        want.step(stop_s=0.0)
        assert np.array_equal(bits(fld.values()), bits(want.values()))
        assert [x.tolist() for x in fld.assignment()] == [x.tolist() for x in want.assignment()]


def test_zero_pairs_leave_the_diagram_and_its_assignment():
    f = NAMED["plain_32"]()
    fld, want = gpu_field(f), gpu_field(f)
    for x in (fld, want):
        x.set_threshold(0.1)
    for _ in range(2):
        for x in (fld, want):
            x.step(stop_s=0.0)
        assert len(fld.zero_pairs()) > 0
        assert gpu_rows(fld.diagram()) == gpu_rows(want.diagram())
        assert [x.tolist() for x in fld.assignment()] == [x.tolist() for x in want.assignment()]
    assert np.array_equal(bits(fld.values()), bits(want.values()))


ALLOC = 16


def _solve(fld, f):
    fld.set_threshold(0.1)
    fld.step(stop_s=0.0)
    v = fld.values()
    loss, grad = fld.loss_and_grad(f)
    return bits(v).tobytes(), gpu_rows(fld.diagram()), loss, grad.tobytes()


def test_every_refused_allocation_is_reported_and_the_field_goes_on():
    """Refuses the n-th device allocation for every n that a field needs: of a new
    field, and of a field whose buffers have to grow.  The call fails with
    TSF_ENOMEM; a diagram small enough for the old buffers and the solve that
    failed then both work."""
    import torch

    import paper_2407_12399_gb300 as tsf
    f = NAMED["plain_32"]()
    small = S.linear_field(f.shape)
    dev, small_dev = torch.from_numpy(f).cuda(), torch.from_numpy(small).cuda()
    want = _solve(gpu_field(f), f)
    want_small = gpu_rows(gpu_field(small).diagram())

    for grown in (False, True):
        refused = 0
        for n in range(1, 1000):
            fld = None
            if grown:
                fld = tsf.Field(small_dev)
                fld.set_threshold(0.1)
                tsf.tsf_set_field(fld._h, dev.data_ptr(), 1)
            tsf.tsf_debug_set(ALLOC, n)
            try:
                fld = fld or tsf.Field(dev)
                _solve(fld, f)
            except tsf.TsfError as e:
                assert e.code == tsf.TSF_ENOMEM
                refused += 1
            finally:
                left = tsf.tsf_debug_set(ALLOC, 0)
            if fld is not None:
                tsf.tsf_set_field(fld._h, small_dev.data_ptr(), 1)
                assert gpu_rows(fld.diagram()) == want_small
                tsf.tsf_set_field(fld._h, dev.data_ptr(), 1)
                assert _solve(fld, f) == want
                fld.close()
            if left > 0:  # fewer than n allocations in all
                break
        assert refused > (40 if grown else 80) and left > 0
