"""The list build's float candidate masks against the double predicate by brute
force: group sizes around a warp and a bucket, boxes so small that pairs wrap
one by one, smoothing lengths up to almost half the box, and box sides whose
squares leave the float range (decided pair by pair in double)."""
import numpy as np
import pytest
import torch

from paper_2511_21921_gb300.solver import Solver

from gpu_util import DT

pytestmark = pytest.mark.gpu


def _brute(x, h, L):
    d = x[:, :, None] - x[:, None, :]
    d = np.where(d > 0.5 * L, d - L, d)
    d = np.where(d < -0.5 * L, d + L, d)
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    g = r2 < (h * h)[:, None]
    s = r2 < (h * h)[None, :]
    np.fill_diagonal(g, False)
    np.fill_diagonal(s, False)
    return g, g | s


def _rows(csr):
    row, col = (t.cpu().numpy() for t in csr)
    return [col[a:b].tolist() for a, b in zip(row[:-1], row[1:])]


@pytest.mark.parametrize("precision,scale", [("mixed", 1.0), ("mixed", 2.5), ("fp64", 1.0),
                                             ("fp64", 2.0 ** 80), ("fp64", 2.0 ** -40)])
@pytest.mark.parametrize("n", [1, 9, 31, 33, 700])
def test_lists_match_the_double_predicate(precision, scale, n):
    rng = np.random.default_rng(n)
    x = rng.random((3, n)) * scale
    x[:, 1::3] = x[:, ::3][:, : x[:, 1::3].shape[1]]  # coincident particles
    h = scale * np.where(rng.random(n) < 0.2, 0.499, 10.0 ** rng.uniform(-3, -0.5, n))
    if precision == "mixed":
        h = h.astype(np.float32).astype(np.float64)
    s = Solver(n, 1, precision, nbr_cap=max(n, 8))
    s.cell_build(torch.tensor(x, device="cuda"),
                 torch.tensor(h, dtype=DT[precision], device="cuda"), L_box=scale)
    g, u = _brute(x, h, scale)
    for mode, want in (("gather", g), ("union", u)):
        got = _rows(s.neighbors_csr(mode))
        assert got == [np.nonzero(r)[0].tolist() for r in want]
