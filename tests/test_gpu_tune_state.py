"""What a tuning run reports and keeps for the sweeps that it did not time: the choice
the plan had, or the rule's variant."""
import pytest
import torch

from paper_2511_21921_gb300 import _lib as L
from paper_2511_21921_gb300 import synth
from paper_2511_21921_gb300.solver import Solver

from gpu_util import to_dev

pytestmark = pytest.mark.gpu

FORWARD, ADJOINT = L.SWEEPS[:4], L.SWEEPS[4:]


def _tuned(s, t, times=1):
    s.cell_build(t["x"], t["h"])
    for _ in range(times):
        out = s.autotune(t["m"], t["v"], t["u"], repeats=1)
    return {k: out[k]["variant"] for k in L.SWEEPS}


def _box(n):
    t = to_dev(synth.lattice(8, seed=1), "mixed")
    return {k: v[..., :n].contiguous() if torch.is_tensor(v) else v for k, v in t.items()}


def test_forward_tuning_keeps_the_adjoint_choices():
    t = _box(512)
    rule = Solver(512, 1, "mixed")
    assert all(_tuned(rule, t, times=2)[k] == 6 for k in ADJOINT)
    s = Solver(512, 1, "mixed")
    s.tune_set([1, 2, 3, 4, 5, 7, 8, 10])
    got = _tuned(s, t)
    assert [got[k] for k in ADJOINT] == [5, 7, 8, 10]


def test_tuning_without_particles_times_nothing():
    t = _box(0)
    s = Solver(512, 1, "mixed")
    assert [_tuned(s, t)[k] for k in L.SWEEPS] == [3, 3, 12, 9, 6, 6, 6, 6]
    s.tune_set([1, 2, 3, 4, 5, 7, 8, 10])
    assert [_tuned(s, t)[k] for k in L.SWEEPS] == [1, 2, 3, 4, 5, 7, 8, 10]
