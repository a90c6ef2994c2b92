"""A sort whose look-back gives up (forced by knob 15: no polls at all) makes the
call that uses it fail with TSF_ETIMEOUT, reads and writes nothing through its
unwritten indices, and leaves the field usable.

The field has 4847 diagram points: sorts of the points rank them by counting
(up to 8192 items) and cannot give up, sorts of two entries per point can."""
import numpy as np
import pytest

from paper_2407_12399_gb300 import synthetic as S

from .test_gpu_parity import NAMED, bits, gpu_field

pytestmark = pytest.mark.gpu

POLLS = 15


def _plain():
    fld = gpu_field(NAMED["plain_32"]())
    fld.set_threshold(0.1)
    assert 4096 < len(fld.diagram()) <= 8192
    return fld


def test_loss_gradient_reports_a_sort_that_gave_up():
    import paper_2407_12399_gb300 as tsf
    f = NAMED["plain_32"]()
    fld = _plain()
    old = tsf.tsf_debug_set(POLLS, -1)
    try:
        with pytest.raises(tsf.TsfError) as e:
            fld.loss_and_grad(f)
    finally:
        tsf.tsf_debug_set(POLLS, old)
    assert e.value.code == tsf.TSF_ETIMEOUT
    loss, grad = fld.loss_and_grad(f)
    want_loss, want = _plain().loss_and_grad(f)
    assert loss == want_loss
    assert np.array_equal(grad.view(np.uint64), want.view(np.uint64)) and np.any(grad)


def test_a_step_reports_a_sort_that_gave_up_and_changes_nothing():
    import paper_2407_12399_gb300 as tsf
    fld = _plain()
    old = tsf.tsf_debug_set(POLLS, -1)
    try:
        with pytest.raises(tsf.TsfError) as e:
            fld.step(stop_s=0.0)
    finally:
        tsf.tsf_debug_set(POLLS, old)
    assert e.value.code == tsf.TSF_ETIMEOUT
    assert np.array_equal(bits(fld.values()), bits(NAMED["plain_32"]()))
    fld.step(stop_s=0.0)
    want = _plain()
    want.step(stop_s=0.0)
    assert np.array_equal(bits(fld.values()), bits(want.values()))
    assert fld.assignment()[0].tolist() == want.assignment()[0].tolist()


# the vertices' order (first diagram), and the still pairs' key orders (more
# points than are ranked by counting)
@pytest.mark.parametrize("shape", [(32, 32, 32), (44, 44, 44)])
def test_diagram_and_matching_report_a_sort_that_gave_up(shape):
    import torch

    import paper_2407_12399_gb300 as tsf
    f = S.random_field(shape, seed=2, kind="uniform")
    dev = torch.from_numpy(f).cuda()
    fld = tsf.Field(dev)
    old = tsf.tsf_debug_set(POLLS, -1)
    try:
        with pytest.raises(tsf.TsfError) as e:
            fld.set_threshold(0.7)
        assert e.value.code == tsf.TSF_ETIMEOUT
    finally:
        tsf.tsf_debug_set(POLLS, old)
    fld.set_threshold(0.7)
    np0 = len(fld.diagram())
    old = tsf.tsf_debug_set(POLLS, -1)
    try:  # the same values: their order is kept, only the matching sorts
        if np0 > 8192:
            with pytest.raises(tsf.TsfError) as e:
                fld.loss_and_grad(f)
            assert e.value.code == tsf.TSF_ETIMEOUT
    finally:
        tsf.tsf_debug_set(POLLS, old)
    loss, grad = fld.loss_and_grad(f)
    other = tsf.Field(dev)
    other.set_threshold(0.7)
    want_loss, want = other.loss_and_grad(f)
    assert loss == want_loss and np.array_equal(grad.view(np.uint64), want.view(np.uint64))
