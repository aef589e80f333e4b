"""The autotuner times the library's own default beside its candidates, whatever
the precision class, so that it never returns something slower than no tuning
(host logic, no GPU)."""
import pytest
import torch

import paper_2607_14054_gb300 as P
from paper_2607_14054_gb300 import autotune as at


class FakePlan:
    carried, extended = False, False

    def __init__(self, lengths, kmax, tuning=None, device=None):
        self.tuning, self.n = tuple(tuning), len(lengths)

    def prepare(self, sos, K):
        pass

    def plan_info(self):
        return torch.full((self.n,), -1 if self.carried else 64), torch.ones(self.n)

    def plan_extended(self):
        return torch.full((self.n,), 2 if self.extended else 0)


@pytest.mark.parametrize("carried", [False, True])
@pytest.mark.parametrize("extended", [False, True])
def test_default_is_timed_and_wins_when_fastest(monkeypatch, carried, extended):
    monkeypatch.setattr(FakePlan, "carried", carried)
    monkeypatch.setattr(FakePlan, "extended", extended)
    monkeypatch.setattr(P, "SosFilter", FakePlan)
    monkeypatch.delenv("SOSFILT_TUNE_CACHE", raising=False)
    timed = []

    def time_apply(plan, *a):
        timed.append(plan.tuning)
        return 1.0 if plan.tuning == (0, 0, 0, 0) else 2.0

    monkeypatch.setattr(at, "_time_apply", time_apply)
    at.clear_cache()
    sos = torch.tensor([[1.0, 0, 0, 1, 0, 0]], dtype=torch.float64)
    assert at.autotune(torch.zeros(100), sos) == (0, 0, 0, 0)
    at.clear_cache()
    assert set(at.candidates(carried, extended)) < set(timed) and len(set(timed)) == len(timed)
