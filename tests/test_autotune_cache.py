"""The autotuner's bookkeeping, without a GPU: the plan's own choice is among the
candidates it times in 2D and 3D, and an entry that other kernels were timed for is not
used."""
import json

import numpy as np
import pytest
import torch

from paper_2110_03345_gb300 import autotune, binding


class FakePlan:
    """Times a step as `cost` says for the options set last."""
    cost = staticmethod(lambda o: 1.0)

    def __init__(self, *a, **k):
        self.opts = {}

    def set_options(self, **o):
        self.opts = o

    def forward(self, *a):
        pass

    gradient = forward

    def stats(self):
        return dict(batch=1, fwd_ms=self.cost(self.opts), adj_ms=0.0)

    def close(self):
        pass


@pytest.fixture
def plan(monkeypatch):
    monkeypatch.setattr(autotune.binding, "Plan", FakePlan)
    return FakePlan


def tune(shape, path, **kw):
    geo = binding.Geometry(np.full((1, 1, len(shape)), 1e-3), np.full((2, len(shape)), 1e-3))
    t = torch.zeros(shape)
    return autotune.tune(shape, 1e-4, 1e-8, 8, 4, 1500.0, t, t, geo, torch.zeros(1, 1, 20),
                         cache_path=str(path), **kw)


@pytest.mark.parametrize("shape", [(32, 40), (16, 20, 24)])
def test_the_plans_own_choice_can_win(plan, monkeypatch, tmp_path, shape):
    monkeypatch.setattr(plan, "cost", staticmethod(lambda o: 0.5 if o["tile"] == 0 else 1.0))
    assert tune(shape, tmp_path / "c.json") == dict(tile=0)


def test_entries_of_other_kernels_are_tuned_again(plan, tmp_path):
    path, shape = tmp_path / "c.json", (16, 20, 24)
    key = autotune.problem_key(shape, 8, True, False, 1)
    for stale in ({}, {"kernels": "0" * 16}):
        path.write_text(json.dumps({key: dict(options=dict(tile=99), ms_per_step=0.0, tried=[], **stale)}))
        assert tune(shape, path, candidates=[dict(tile=7)]) == dict(tile=7)
    assert tune(shape, path, candidates=[]) == dict(tile=7)      # the new entry stands
    assert tune(shape, path, candidates=[dict(tile=8)], refresh=True) == dict(tile=8)
    assert json.loads(path.read_text())[key]["kernels"] == autotune.kernels_id()
