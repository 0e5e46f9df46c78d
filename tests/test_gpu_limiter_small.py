"""The velocity-gradient limiter at the lower end of the range: a smooth velocity
field decays over many decades, and the limiter, a function of the ratio of two
projected gradients, has to stay finite and right where their powers leave the range
of normal numbers."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import TOL, rel_l2, run_forward, to_dev

pytestmark = pytest.mark.gpu


def _decaying(width):
    """Velocities exp(-(r/width)^2) around the middle of the box."""
    d = synth.lattice(16, seed=5)
    r2 = ((d["x"] - 0.5) ** 2).sum(0)
    d["v"] = np.exp(-r2 / width ** 2) * np.array([1.0, 0.7, -0.4])[:, None]
    return d


# fp64, 1/45 of the side: 486 pairs whose projected gradients have the same sign and a
# sum below 7.5e-155, the square root of the smallest normal double's neighborhood
@pytest.mark.parametrize("precision,width", [("fp64", 1 / 45.0), ("fp64", 1 / 30.0),
                                             ("mixed", 1 / 9.0), ("mixed", 1 / 7.0)])
def test_rates_of_a_decaying_velocity_field(precision, width):
    d = _decaying(width)
    ref = oracle.forward(d["x"], d["h"], d["m"], d["v"], d["u"], 1.0, want=("dvdt", "dudt"))
    got, _ = run_forward(d, precision)
    for k in ("dvdt", "dudt"):
        assert np.isfinite(got[k]).all(), k
        assert rel_l2(got[k], ref[k]) <= TOL[precision], k


# every pair's projected gradients so small that the cube of their sum is no normal
# number; the derivative of the limiter itself is of ordinary size there
@pytest.mark.parametrize("precision,scale,tol", [("fp64", 1e-120, 1e-10), ("fp64", 1e-140, 1e-10),
                                                 ("mixed", 1e-13, 2e-4), ("mixed", 1e-14, 2e-4)])
@pytest.mark.parametrize("which", ["x", "v"])
def test_gradient_of_small_velocities(precision, scale, tol, which):
    d = synth.lattice(12, seed=6)
    d["v"] = d["v"] * scale
    n = d["h"].shape[0]
    ga, gu = synth.cotangents(n, seed=4)
    t = to_dev(d, precision)
    s = Solver(n, 1, precision)
    s.cell_build(t["x"], t["h"])
    s.moments(t["m"])
    s.rates(t["v"], t["u"])
    g = s.adjoint(t["v"], t["u"], torch.tensor(ga, dtype=s.dtype, device="cuda"),
                  torch.tensor(gu, dtype=s.dtype, device="cuda"), recompute=False)
    g = [a.double().cpu().numpy() for a in g]
    assert all(np.isfinite(a).all() for a in g)
    k = "xv".index(which)
    tan = np.random.default_rng(11).normal(size=(3, n))
    _, out = oracle.jvp(d["x"], d["h"], d["m"], d["v"], d["u"], d["L"], **{"t" + which: tan},
                        want=("dvdt", "dudt"))
    lhs = (ga * out["dvdt"]).sum() + (gu * out["dudt"]).sum()
    assert abs(lhs - (g[k] * tan).sum()) <= tol * np.abs(g[k] * tan).sum()


@pytest.mark.parametrize("precision,width", [("fp64", 1 / 45.0), ("fp64", 1 / 30.0),
                                             ("mixed", 1 / 9.0), ("mixed", 1 / 7.0)])
def test_gradient_of_a_decaying_velocity_field_is_finite(precision, width):
    d = _decaying(width)
    n = d["h"].shape[0]
    ga, gu = synth.cotangents(n, seed=3)
    t = to_dev(d, precision)
    s = Solver(n, 1, precision)
    s.cell_build(t["x"], t["h"])
    s.moments(t["m"])
    s.rates(t["v"], t["u"])
    for a in s.adjoint(t["v"], t["u"], torch.tensor(ga, dtype=s.dtype, device="cuda"),
                       torch.tensor(gu, dtype=s.dtype, device="cuda"), recompute=False):
        assert torch.isfinite(a).all()
