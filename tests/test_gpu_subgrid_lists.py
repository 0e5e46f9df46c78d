"""Subgrid sums whose bucket list is empty, partly filled, just full or has to be
emptied on the way (160 buckets of eight gas particles), against brute force."""
import numpy as np
import pytest
import torch

from oracle import subgrid as S
from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import DT, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("side", [2, 12, 20])
def test_bucket_lists_of_every_length(precision, tol, side):
    d = synth.lattice(side, seed=3, k_target=40)
    n = side ** 3
    rng = np.random.default_rng(side)
    if side == 2:
        d["h"][:] = 0.45
    else:
        d["h"][::50] = 0.45  # scatter reach across the box: every bucket is listed
    n_s = 24
    xs = rng.random((3, n_s))
    hs = np.linspace(0.01, 0.49, n_s)
    q = rng.uniform(0.1, 1.0, (3, n_s))
    if precision == "mixed":
        d["h"], hs, q = (a.astype(np.float32).astype(np.float64) for a in (d["h"], hs, q))
    t = to_dev(d, precision)
    s = Solver(n, 1, precision, nbr_cap=n + 32)
    s.cell_build(t["x"], t["h"])
    Vg, _ = s.moments(t["m"], want_V=True)
    x_d = torch.tensor(xs, device="cuda")
    h_d = torch.tensor(hs, dtype=DT[precision], device="cuda")
    V, hv = s.subgrid_volume(x_d, h_d, n_h=2.25)
    dq, A = s.subgrid_deposit(x_d, h_d, torch.tensor(q, dtype=DT[precision], device="cuda"))
    eV, eh = S.volume(xs, hs, d["x"], d["h"], n_h=2.25)
    edq, eA = S.deposit(xs, hs, q, d["x"], Vg.double().cpu().numpy())
    for got, want in ((V, eV), (hv, eh), (A, eA), (dq, edq)):
        g = got.double().cpu().numpy()
        assert np.linalg.norm(g - want) <= tol * np.linalg.norm(want)
