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


@pytest.mark.parametrize("n", [1023, 1024, 1025, 2049, 155648, 155649, 311297, 622592, 622593])
def test_pairs_at_the_sort_tile_edges(n):
    """Sizes where the sort's tiles or its dispatch change, several boxes of two
    sides: the number of pairs and the lists of sampled particles from a k-d tree."""
    from scipy.spatial import cKDTree
    rng = np.random.default_rng(n)
    off = np.array([0, n // 3, n // 3, n], np.int64)  # the middle box is empty
    side = np.array([1.0, 1.0, 2.5])
    x, h = np.empty((3, n)), np.empty(n)
    total = 0
    rows = {}
    for b in range(3):
        a, e = off[b], off[b + 1]
        if e == a:
            continue
        x[:, a:e] = rng.random((3, e - a)) * side[b]
        hb = np.float32(1.2 * side[b] * (e - a) ** (-1 / 3) if e - a > 27 else 0.3 * side[b])
        h[a:e] = hb
        t = cKDTree(x[:, a:e].T, boxsize=side[b])
        total += t.count_neighbors(t, float(hb)) - (e - a)
        for i in rng.integers(0, e - a, 20):
            rows[a + i] = sorted(a + k for k in t.query_ball_point(x[:, a + i], float(hb)) if k != i)
    s = Solver(n, 3, "mixed")
    s.cell_build(torch.tensor(x, device="cuda"), torch.tensor(h, dtype=torch.float32, device="cuda"),
                 box_off=torch.tensor(off, device="cuda"), box_L=torch.tensor(side, device="cuda"))
    assert s.stats()["gather_pairs"] == s.stats()["union_pairs"] == total
    row, col = (t.cpu().numpy() for t in s.neighbors_csr("gather"))
    for i, want in rows.items():
        assert col[row[i]:row[i + 1]].tolist() == want
