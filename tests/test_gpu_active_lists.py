"""Compacted lists of the active-set evaluation at sizes around a warp, a block and
the tiles that are counted: the particles written are those flagged, each with the
values of the whole evaluation."""
import numpy as np
import pytest
import torch

from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 2047, 2048, 2049, 4097, 12167])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_flagged_particles_and_no_others(n, share):
    d = synth.lognormal(23, 1.0, seed=2)
    keep = np.random.default_rng(n).permutation(d["h"].shape[0])[:n]
    d = {k: (v[..., keep] if isinstance(v, np.ndarray) and v.shape[-1:] == (12167,) else v)
         for k, v in d.items()}
    t = to_dev(d, "mixed")
    s = Solver(n, 1, "mixed")
    s.cell_build(t["x"], t["h"])
    V, C = s.moments(t["m"], want_V=True, want_coef=True)
    V, C = V.clone(), C.clone()
    rng = np.random.default_rng(7 * n + 1)
    f = (rng.random(n) < share) * 1 + (rng.random(n) < 0.5 * share) * 2
    flags = torch.tensor(f, dtype=torch.uint8, device="cuda")
    V2, C2 = torch.full_like(V, 3.0), torch.full_like(C, 3.0)
    s.moments_active(t["m"], flags, V2, C2)
    re = flags != 0
    assert torch.equal(V2[re], V[re]) and bool((V2[~re] == 3.0).all())
    assert bool((C2[:, ~re] == 3.0).all())
    # the volumes of particles that keep theirs enter the others' coefficients
    V3, C3 = V.clone(), C.clone()
    s.moments_active(t["m"], flags, V3, C3)
    assert torch.equal(V3, V) and torch.equal(C3.nan_to_num(), C.nan_to_num())
