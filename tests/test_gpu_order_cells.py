"""The merged vertex order with few to many changed values (the edges of its
32-key rank blocks, its limit and past it), and the critical-cell lists and D1
candidates of fields whose vertex count ends at, before and after the
2048-vertex tiles of the two passes that write them."""
import numpy as np
import pytest

import oracle
import paper_2407_12399_gb300 as tsf
from paper_2407_12399_gb300 import synthetic as S

from .test_gpu_parity import gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("changed", [0, 1, 31, 32, 33, 255, 257, 4097, tsf.INCREMENTAL_ORDER_MAX,
                                     tsf.INCREMENTAL_ORDER_MAX + 1])
def test_merged_order_gives_the_diagram_of_a_new_field(changed):
    f = S.random_field((31, 33, 35), seed=changed, kind="uniform")
    fld = gpu_field(f)
    fld.set_threshold(0.95)  # few targets: the matching is not what is tested
    rng = np.random.default_rng(changed)
    at = rng.permutation(f.size)[:changed]
    for k in range(2):  # twice: the second from a merged order
        f = f.copy()
        f.ravel()[at] = rng.choice(f.ravel(), changed) + np.float32(0.25 * k - 0.5)
        fld.loss_and_grad(f)
        assert gpu_rows(fld.diagram()) == gpu_rows(gpu_field(f).diagram())


@pytest.mark.parametrize("part", [1 / 16 - 1e-5, 1 / 16 + 1e-5, 1.0], ids=["listed", "marked", "all"])
def test_lower_stars_after_many_changes(part):
    """Changes on either side of a sixteenth of a grid large enough for marks
    instead of a list; its size is no multiple of the 512-vertex windows."""
    f = S.random_field((79, 81, 83), seed=5, kind="uniform")
    fld = gpu_field(f)
    fld.set_threshold(0.98)
    rng = np.random.default_rng(6)
    for _ in range(2):
        at = rng.permutation(f.size)[:int(part * f.size)]
        f = f.copy()
        f.ravel()[at] = rng.uniform(0, 1, len(at))
        fld.loss_and_grad(f)
        a, b = fld.diagram(), gpu_field(f).diagram()
        assert len(a) == len(b) and all(np.array_equal(a[k], b[k]) for k in a.dtype.names)


@pytest.mark.parametrize("shape", [(2, 2, 511), (2, 32, 32), (3, 3, 228), (2, 2, 513), (4, 23, 89), (2, 2048, 2),
                                   (5, 7, 117), (27, 27, 27)])
@pytest.mark.parametrize("kind", ["uniform", "ties"])
def test_cells_at_tile_ends(shape, kind):
    f = S.random_field(shape, seed=sum(shape), kind=kind)
    assert gpu_rows(gpu_field(f).diagram()) == oracle_rows(f, oracle.diagram(f)["pairs"])
