"""The active-set evaluation writes every flagged particle, at sizes around a warp, a
block and the tiles whose flags are counted: what it has to write holds another value
before each call."""
import numpy as np
import pytest
import torch

from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import to_dev

pytestmark = pytest.mark.gpu

POISON = 3.0


def _same(a, b):
    return torch.equal(a.nan_to_num(), b.nan_to_num())


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 2047, 2048, 2049, 4097, 12167])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_every_flagged_particle_is_written(n, share):
    d = synth.lognormal(23, 1.0, seed=2)
    keep = np.random.default_rng(n).permutation(d["h"].shape[0])[:n]
    d = {k: (v[..., keep] if isinstance(v, np.ndarray) and v.shape[-1:] == (12167,) else v)
         for k, v in d.items()}
    t = to_dev(d, "mixed")
    s = Solver(n, 1, "mixed")
    s.cell_build(t["x"], t["h"])
    V, C = s.moments(t["m"], want_V=True, want_coef=True)
    dv, du, rho, gv = s.rates(t["v"], t["u"], want_rho=True, want_gradv=True)
    rng = np.random.default_rng(7 * n + 1)
    f = (rng.random(n) < share) * 1 + (rng.random(n) < 0.5 * share) * 2
    flags = torch.tensor(f, dtype=torch.uint8, device="cuda")
    re, act = flags != 0, (flags & 1) != 0
    # stored fields of the others, poison where the call has to write
    V2, C2, rho2, gv2 = (a.clone() for a in (V, C, rho, gv))
    V2[re], C2[:, re] = POISON, POISON
    s.moments_active(t["m"], flags, V2, C2)
    assert _same(V2, V) and _same(C2, C)
    rho2[act], gv2[:, act] = POISON, POISON
    out = (torch.full_like(dv, POISON), torch.full_like(du, POISON))
    s.rates_active(t["v"], t["u"], rho2, gv2, out=out)
    assert _same(rho2, rho) and _same(gv2, gv)
    assert _same(out[0][:, act], dv[:, act]) and _same(out[1][act], du[act])
    assert bool((out[0][:, ~act] == POISON).all()) and bool((out[1][~act] == POISON).all())
