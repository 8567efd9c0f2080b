"""AcrlStep.run's choice between one call and the two halves, on an object whose buffers are host tensors."""

from types import SimpleNamespace

import pytest
import torch

import paper_2607_24062_gb300 as acrl
from paper_2607_24062_gb300 import pipeline

T, S, GN = 6, 2, 1


def _step(cls=acrl.AcrlStep):
    step = object.__new__(cls)
    step.T, step.V, step.S, step.Gn, step.params = T, 8, S, GN, acrl.Params()
    step.logp = torch.empty(T)
    step.disc = SimpleNamespace(S=S, Gn=GN)
    for name in ("state", "lse", "entropy", "adv", "weight", "coef", "alpha", "ent_coef", "grad", "token_loss", "loss", "flags"):
        setattr(step, name, None)
    return step


def _args():
    return (torch.empty(T, 8), None, None, None, torch.empty(S), torch.empty(S + 1), torch.empty(GN + 1))


@pytest.fixture
def calls(monkeypatch):
    made = []
    monkeypatch.setattr(pipeline.api, "step", lambda *a, **kw: made.append("step"))
    for name in ("token_stats", "seq_discrepancy", "grpo_advantage", "controller_step", "loss_grad_logits"):
        monkeypatch.setattr(pipeline.api, name, lambda *a, _n=name, **kw: made.append(_n))
    return made


def test_one_call(calls):
    _step().run(*_args())
    assert calls == ["step"]


@pytest.mark.parametrize("name", ["statistics", "gradient"])
@pytest.mark.parametrize("where", ["object", "subclass", "class", "another object"])
def test_an_overridden_half_is_called(calls, monkeypatch, name, where):
    def mine(*a, **kw):
        calls.append("mine")

    step = _step()
    if where == "object":
        setattr(step, name, mine)
    elif where == "another object":
        other = _step(type("Other", (acrl.AcrlStep,), {name: mine}))
        setattr(step, name, getattr(other, name))
    elif where == "subclass":
        step = _step(type("Mine", (acrl.AcrlStep,), {name: mine}))
    else:
        monkeypatch.setattr(acrl.AcrlStep, name, mine)
    step.run(*_args())
    assert "mine" in calls and "step" not in calls


@pytest.mark.parametrize("so,go", [(0, 2), (3, 0)])
def test_weights_refuse_empty_offsets(so, go):
    with pytest.raises(acrl.AcrlError):
        acrl.importance_weights(torch.zeros(48, dtype=torch.uint8), acrl.Params(), torch.zeros(4), torch.zeros(4), None,
                                torch.zeros(2), torch.zeros(so, dtype=torch.int64), torch.zeros(go, dtype=torch.int32))
