"""Staging of the list build: buckets in fours and eights, the ring of three stages
and buckets that hold particles of two boxes, at counts around a bucket, a stage
and the ring."""
import numpy as np
import pytest
import torch

from paper_2511_21921_gb300.solver import Solver

pytestmark = pytest.mark.gpu


def _rows(csr):
    row, col = (t.cpu().numpy() for t in csr)
    return [col[a:b].tolist() for a, b in zip(row[:-1], row[1:])]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("sizes", [(31,), (32,), (63,), (65,), (95,), (97,), (129,), (257,),
                                   (3, 5), (29, 6, 60), (1, 96, 7, 100), (13,) * 20])
def test_dense_boxes_of_ragged_sizes(precision, sizes):
    n = sum(sizes)
    rng = np.random.default_rng(n)
    off = np.concatenate([[0], np.cumsum(sizes)])
    x, h = rng.random((3, n)), 0.45 * (0.3 + 0.7 * rng.random(n))
    s = Solver(n, len(sizes), precision, nbr_cap=max(sizes))
    s.cell_build(torch.tensor(x, device="cuda"),
                 torch.tensor(h, dtype=s.dtype, device="cuda"),
                 box_off=torch.tensor(off, device="cuda"),
                 box_L=torch.ones(len(sizes), dtype=torch.float64, device="cuda"))
    if precision == "mixed":
        h = h.astype(np.float32).astype(np.float64)
    d = np.abs(x[:, :, None] - x[:, None, :])
    d = np.minimum(d, 1.0 - d)
    r2 = (d * d).sum(0)
    box = np.repeat(np.arange(len(sizes)), sizes)
    pair = (box[:, None] == box[None, :]) & ~np.eye(n, dtype=bool)
    g = pair & (r2 < (h * h)[:, None])
    u = pair & ((r2 < (h * h)[:, None]) | (r2 < (h * h)[None, :]))
    for mode, want in (("gather", g), ("union", u)):
        assert _rows(s.neighbors_csr(mode)) == [np.nonzero(r)[0].tolist() for r in want]
