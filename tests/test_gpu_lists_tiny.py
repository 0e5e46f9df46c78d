"""Neighbor lists for smoothing lengths so small that their squares, and the rounding
band of the float candidate test, leave the range of normal floats: the lists are
still those of the double predicate."""
import numpy as np
import pytest
import torch

from paper_2511_21921_gb300.solver import Solver

from gpu_util import DT

pytestmark = pytest.mark.gpu


def _rows(csr):
    row, col = (t.cpu().numpy() for t in csr)
    return [col[a:b].tolist() for a, b in zip(row[:-1], row[1:])]


# box side and the decades of h: just above and below 1e-33 of a unit box, where the
# band's product with the side leaves the range; a small box, where it does so earlier;
# smoothing lengths of the FP64 form below every float
@pytest.mark.parametrize("precision,L,lo,hi", [("mixed", 1.0, -36, -28), ("fp64", 1.0, -36, -28),
                                               ("mixed", 2e-6, -37, -28), ("fp64", 2e-6, -37, -28),
                                               ("fp64", 1.0, -120, -40)])
@pytest.mark.parametrize("where", ["coincident", "origin"])
def test_lists_of_tiny_smoothing_lengths(precision, L, lo, hi, where):
    n = 200
    rng = np.random.default_rng(4)
    h = 10.0 ** rng.uniform(lo, hi, n)
    if where == "coincident":
        x = rng.random((3, n)) * L
        x[:, 1::2] = x[:, ::2]
        h[: n // 4] = 10.0 ** lo
    else:  # around the origin, as far apart as they reach
        x = 10.0 ** rng.uniform(lo, hi, n) * rng.random((3, n))
    if precision == "mixed":
        h = h.astype(np.float32).astype(np.float64)
    s = Solver(n, 1, precision, nbr_cap=n)
    s.cell_build(torch.tensor(x, device="cuda"),
                 torch.tensor(h, dtype=DT[precision], device="cuda"), L_box=L)
    d = x[:, :, None] - x[:, None, :]
    d = np.where(d > 0.5 * L, d - L, np.where(d < -0.5 * L, d + L, d))
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    other = ~np.eye(n, dtype=bool)
    g = other & (r2 < (h * h)[:, None])
    u = g | (other & (r2 < (h * h)[None, :]))
    for mode, want in (("gather", g), ("union", u)):
        assert _rows(s.neighbors_csr(mode)) == [np.nonzero(r)[0].tolist() for r in want]
