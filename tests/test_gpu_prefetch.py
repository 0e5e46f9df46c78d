"""Prefetch distances of the plain loads, up to more entries than a list has: a hint
that changes no result."""
import pytest
import torch

from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _rates(t, variant, **params):
    n = t["h"].shape[0]
    s = Solver(n, 1, "mixed", **params)
    s.tune_set([variant] * 8)
    s.cell_build(t["x"], t["h"])
    s.moments(t["m"])
    dv, du, _, _ = s.rates(t["v"], t["u"])
    g = s.adjoint(t["v"], t["u"], torch.ones_like(dv), torch.ones_like(du), recompute=False)
    assert s.poll() in (0, 6)  # 6: a particle with so few neighbors that its moment is singular
    return dv, du, *g


@pytest.mark.parametrize("distance", [1, 3, 16])
@pytest.mark.parametrize("variant", [0, 2])
def test_distances_change_no_bit(distance, variant):
    t = to_dev(synth.lognormal(11, 1.0, seed=8), "mixed")
    t["h"][::7] *= 0.2  # short lists
    for a, b in zip(_rates(t, variant), _rates(t, variant, prefetch=distance)):
        assert torch.equal(a.nan_to_num(), b.nan_to_num())
