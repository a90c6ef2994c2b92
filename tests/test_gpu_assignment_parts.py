"""Reduced assignments of diagrams large enough for the split candidate scan
(2^14 points and more) and, next to them, smaller ones: the matching and the
trajectory of the oracle, step by step, with free targets in several groups;
points sorted by rank counting (few) and by radix sorts (many)."""
import numpy as np
import pytest

import oracle
from paper_2407_12399_gb300 import synthetic as S

from .test_gpu_parity import bits, gpu_field

pytestmark = pytest.mark.gpu

CASES = {
    "split_noise": (lambda: S.gaussian_mixture((46, 47, 48), n_bumps=8, seed=5, noise_frac=0.3), 0.15),
    "split_ties": (lambda: (np.round(S.gaussian_mixture((50, 47, 48), n_bumps=8, seed=6, noise_frac=0.2) * 63) /
                            63).astype(np.float32), 0.2),
    "few_points": (lambda: S.gaussian_mixture((21, 22, 23), n_bumps=6, seed=7, noise_frac=0.3), 0.1),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_assignments_and_trajectory_match_the_oracle(name):
    make, tau = CASES[name]
    f0 = make()
    fld = gpu_field(f0)
    fld.set_threshold(tau)
    ref = oracle.Solver(f0, tau=tau)
    seen = 0
    for j in range(3):
        tgt, still = fld.assignment()
        P = ref.points()
        assert tgt.tolist() == P["tgt"].tolist(), f"assignment differs at j={j}"
        assert still.tolist() == P["still"].tolist()
        if name.startswith("split"):
            assert len(tgt) >= 1 << 14
        seen += fld.step(stop_s=0.0)["n_nonstill_matched"]
        ref.iterate(stop_s=0.0)
        assert np.array_equal(bits(fld.values()), bits(ref.field())), f"field differs after step {j + 1}"
    assert seen > 0, "no free target was matched: the case does not reach the candidate scan"
