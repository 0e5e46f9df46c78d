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

from gpu_util import TOL, rel_l2, run_forward

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
