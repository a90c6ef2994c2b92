"""A sort whose look-back gives up (forced by knob 15: no polls at all) makes the
call that uses it fail with TSF_ETIMEOUT, reads and writes nothing through its
unwritten indices, and leaves the field usable.

The field has 4847 diagram points: sorts of the points rank them by counting
(up to 8192 items) and cannot give up, sorts of two entries per point can."""
import numpy as np
import pytest

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
