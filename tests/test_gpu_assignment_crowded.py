"""Crowded assignments: more free targets in a group than a candidate tile holds,
so the general path's buffers grow to what the first call needs."""
import numpy as np
import pytest

from paper_2407_12399_gb300 import synthetic as S

from .test_gpu_parity import gpu_field

pytestmark = pytest.mark.gpu


def test_first_crowded_matching_is_complete():
    """At the values the targets were taken from, the optimal matching gives
    every target its own point, so the loss is the initial one: the diagonal
    costs of the other points (1363 targets, 6632 points)."""
    import paper_2407_12399_gb300 as tsf
    f = S.random_field((28, 28, 28), seed=2, kind="uniform")
    fld = gpu_field(f)
    fld.set_threshold(0.3)
    loss0 = tsf.tsf_simplify(fld._h, tsf.params(max_iters=0), None, 0).loss0
    nt = len(fld.targets())
    assert nt > 1024
    loss, grad = fld.loss_and_grad(f)
    tgt, _ = fld.assignment()
    matched = tgt[tgt >= 0]
    assert sorted(matched.tolist()) == list(range(nt))
    assert loss == loss0
    d, t = fld.diagram(), fld.targets()
    own = np.flatnonzero(tgt >= 0)
    for key in ("dim", "v_birth", "v_death"):
        assert np.array_equal(d[key][own], t[key][matched])
    moved = np.unique(np.concatenate([d["v_birth"][tgt < 0], d["v_death"][tgt < 0]]))
    assert np.count_nonzero(grad) <= len(moved)


def test_crowded_auction_is_within_its_precision_of_the_exact_matching():
    """The same step from the same values, every point matched anew: the auction's
    distance (the square root of the loss) within 1 % of the exact one, and on its
    first call, before any buffer has grown."""
    f = S.random_field((28, 28, 28), seed=2, kind="uniform")
    loss = {}
    for precision in (0.01, 0.0):
        fld = gpu_field(f)
        fld.set_threshold(0.3)
        loss[precision] = fld.step(stop_s=0.0, fast_assignment_update=0, assignment_precision=precision)["loss"]
        tgt, still = fld.assignment()
        assert not still.any()
        matched = tgt[tgt >= 0]
        assert len(np.unique(matched)) == len(matched) > 1024
    assert loss[0.0] <= loss[0.01] * (1 + 1e-12)
    assert np.sqrt(loss[0.01]) <= 1.01 * np.sqrt(loss[0.0])
