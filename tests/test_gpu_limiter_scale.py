"""The limiter's reciprocals at the upper end of the float range: the path has no
unit of its own, so lengths and velocities in units of powers of two have to give
the same bits times powers of two, also where the square and the cube of the
projected gradients' sum come close to the largest float."""
import math

import numpy as np
import pytest
import torch

from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import to_dev

pytestmark = pytest.mark.gpu

LEN = 12  # lengths in units of 2^-LEN


def _pass(t, n, L, ga):
    s = Solver(n, 1, "mixed")
    s.cell_build(t["x"], t["h"], L_box=L)
    s.moments(t["m"])
    dv, du, _, gradv = s.rates(t["v"], t["u"], want_gradv=True)
    g = s.adjoint(t["v"], t["u"], ga, torch.zeros_like(t["u"]), recompute=False)
    row, col = s.neighbors_csr("union")
    assert s.poll() == 0
    return dv, du, gradv, g, row, col


# log2 of the largest sum: just inside the cube's range (42.67 and up overflow), and
# the square's, where only the rates are compared
@pytest.mark.parametrize("top,cubes", [(40.9, True), (42.6, True), (62.0, False)])
def test_powers_of_two_in_the_units_change_no_bit(top, cubes):
    d = synth.lognormal(12, 1.0, seed=3)
    n = d["h"].shape[0]
    t = to_dev(d, "mixed")
    ga = torch.tensor(np.random.default_rng(1).normal(size=(3, n)), dtype=torch.float32,
                      device="cuda")
    dv, du, gradv, g, row, col = _pass(t, n, 1.0, ga)
    i = torch.repeat_interleave(torch.arange(n, device="cuda"), row[1:] - row[:-1])
    j = col.long()
    sep = t["x"][:, i] - t["x"][:, j]
    sep -= torch.round(sep)
    G = gradv.double().view(3, 3, n)
    sums = torch.einsum("ap,abp,bp->p", sep, G[:, :, i] + G[:, :, j], sep).abs()
    k = math.floor(top - LEN - math.log2(sums.max().item()))
    s = {"x": t["x"] * 2.0 ** LEN, "h": t["h"] * 2.0 ** LEN, "m": t["m"],
         "v": t["v"] * 2.0 ** k, "u": t["u"] * 2.0 ** (2 * k)}
    dv2, du2, gradv2, g2, _, _ = _pass(s, n, 2.0 ** LEN, ga * 2.0 ** (LEN - 2 * k))
    assert torch.equal(gradv2, gradv * 2.0 ** (k - LEN))
    assert torch.equal(dv2, dv * 2.0 ** (2 * k - LEN))
    if cubes:
        assert torch.equal(du2, du * 2.0 ** (3 * k - LEN))
        for a, b, e in zip(g2, g, (-LEN, -k, -2 * k, -LEN)):
            assert torch.equal(a, b * 2.0 ** e)
