"""Elder-rule pairs (D0, D2) from the union-find without rounds, on fields whose
merge trees are as deep or as wide as they can be: a staircase of minima along
a serpentine (every component merges into the next older one, and the other
way round), plateaus, and more items than threads in flight.  The pairs are
those of the oracle's plain reduction."""
import numpy as np
import pytest

import oracle

from .test_gpu_parity import gpu_field, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu


def _staircase(shape, down):
    """Isolated extrema along a serpentine, each with the next as its only
    near neighbour, values falling or rising along it."""
    lz, ly, lx = shape
    f = np.zeros(shape, np.float64)
    k = 0
    n = (lz + 1) // 2 * ((ly + 1) // 2) * ((lx + 1) // 2)
    z, y, x = np.meshgrid(np.arange(lz), np.arange(ly), np.arange(lx), indexing="ij")
    f += 2.0 + 1e-3 * (x + lx * (y + ly * z)) / f.size
    for iz in range(0, lz, 2):
        for iy in (range(0, ly, 2) if iz % 4 == 0 else range((ly - 1) // 2 * 2, -1, -2)):
            for ix in (range(0, lx, 2) if iy % 4 == 0 else range((lx - 1) // 2 * 2, -1, -2)):
                f[iz, iy, ix] = (n - k if down else k) / n
                k += 1
    return f.astype(np.float32)


CASES = {
    "falling": lambda: _staircase((11, 21, 31), True),
    "rising": lambda: _staircase((11, 21, 31), False),
    "falling_peaks": lambda: -_staircase((11, 21, 31), True),
    "rising_peaks": lambda: -_staircase((11, 21, 31), False),
    "ties": lambda: np.random.default_rng(3).integers(0, 3, (24, 25, 26)).astype(np.float32),
    "noise": lambda: np.random.default_rng(4).uniform(0, 1, (40, 41, 42)).astype(np.float32),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_elder_rule_pairs_match_the_oracle(name):
    f = CASES[name]()
    assert gpu_rows(gpu_field(f).diagram()) == oracle_rows(f, oracle.diagram(f)["pairs"])
