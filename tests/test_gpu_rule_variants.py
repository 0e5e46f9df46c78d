"""The launch variants an untuned plan takes give the bits of plain loads, on both
sides of the sizes where the rule changes them."""
import pytest
import torch

from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _all(t, choice):
    n = t["h"].shape[0]
    s = Solver(n, 1, "mixed")
    if choice is not None:
        s.tune_set(choice)
    s.cell_build(t["x"], t["h"])
    V, C = s.moments(t["m"], want_V=True, want_coef=True)
    dv, du, rho, gradv = s.rates(t["v"], t["u"], want_rho=True, want_gradv=True)
    ga, gu = torch.sin(10.0 * t["v"]), torch.cos(t["u"])
    g = s.adjoint(t["v"], t["u"], ga, gu, recompute=False)
    f = s.rates_adjoint(t["v"], t["u"], ga, gu)
    return V, C, dv, du, rho, gradv, *g, *f


# the rule's lines are at 50,000 (volume) and 100,000 particles (moments)
@pytest.mark.parametrize("side,n", [(16, 4091), (37, 49999), (37, 50653), (47, 99999),
                                    (47, 103823)])
def test_rule_variants_give_the_bits_of_plain_loads(side, n):
    d = synth.lognormal(side, 1.5, seed=12)
    t = {k: v[..., :n].contiguous() for k, v in to_dev(d, "mixed").items()}
    for a, b in zip(_all(t, None), _all(t, [0] * 8)):
        assert torch.equal(a.nan_to_num(), b.nan_to_num())
