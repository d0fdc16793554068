"""What ActionExpert.step refuses, without a GPU: the library call is replaced by one that records."""
import types

import pytest
import torch

from paper_2607_14695_b200 import binding as rb
from paper_2607_14695_b200 import expert as ex
from paper_2607_14695_b200 import synth

W = synth.CONFIGS["cfg2"].with_(B=2, L=2, T=8, D=64, Hq=2, Hkv=1, d=32, Cd=8, Hd=8, A=8)
F = 64


def _model(cache=None, **weights):
    desc = rb.CacheDesc(W.L, W.B, W.Hq, W.Hkv, W.d, 16, 4, W.T, W.dtype, 1)
    for n, v in (cache or {}).items():
        setattr(desc, n, v)
    m = ex.ActionExpert(W, types.SimpleNamespace(desc=desc), {}, F, device="cpu")
    m.W = {n: torch.zeros(s, dtype=torch.bfloat16) for n, s in m.shapes.items()}
    m.W.update(weights)
    return m


@pytest.fixture
def calls(monkeypatch):
    seen = []
    monkeypatch.setattr(rb, "reflex_expert_step", lambda cache, d, a, cond, k, K, stream=None: seen.append(d) or a)
    return seen


CHUNK, COND = (W.B, W.T, W.A), (W.B, W.Cd)


def test_step_passes_on_what_fits(calls):
    a = torch.zeros(CHUNK)
    assert _model().step(a, torch.zeros(COND, dtype=torch.bfloat16), 0) is a
    assert _model(cache=dict(L=7)).step(a, torch.zeros(COND, dtype=torch.bfloat16), 0) is a
    assert [d.L for d in calls] == [W.L, W.L] and calls[0].F == F
    m = _model()
    m.W.update(b1=m.W["b1"].reshape(-1), Wo=torch.cat([m.W["Wo"]] * 2))
    assert m.step(a, torch.zeros(COND, dtype=torch.bfloat16), 0) is a


@pytest.mark.parametrize("a", [torch.zeros(1, W.T, W.A), torch.zeros(W.B, W.T - 1, W.A), torch.zeros(W.B * W.T, W.A), torch.zeros(CHUNK, dtype=torch.bfloat16),
                               torch.zeros(CHUNK, dtype=torch.float64), torch.zeros(CHUNK, device="meta")], ids=lambda t: f"{list(t.shape)}{t.dtype}{t.device}")
def test_step_refuses_a_chunk_of_another_form(calls, a):
    with pytest.raises(ValueError):
        _model().step(a, torch.zeros(COND, dtype=torch.bfloat16), 0)
    assert not calls


@pytest.mark.parametrize("cond", [torch.zeros(COND), torch.zeros((1, W.Cd), dtype=torch.bfloat16), torch.zeros((W.B, W.Cd + 8), dtype=torch.bfloat16)],
                         ids=lambda t: f"{list(t.shape)}{t.dtype}")
def test_step_refuses_conditioning_of_another_form(calls, cond):
    with pytest.raises(ValueError):
        _model().step(torch.zeros(CHUNK), cond, 0)
    assert not calls


@pytest.mark.parametrize("name", ex._WEIGHTS)
def test_step_refuses_weights_of_another_form(calls, name):
    good = _model().W[name]
    for bad in (good.float(), good[:1] if name in ex._LAYERS else torch.zeros((good.shape[0] + 1,) + tuple(good.shape[1:]), dtype=good.dtype), good[..., :-1].contiguous()):
        with pytest.raises(ValueError, match=name):
            _model(**{name: bad}).step(torch.zeros(CHUNK), torch.zeros(COND, dtype=torch.bfloat16), 0)
    assert not calls


@pytest.mark.parametrize("cache", [dict(B=3), dict(B=1), dict(L=1), dict(Hq=4), dict(Hkv=2), dict(d=64), dict(dtype=synth.DTYPE_F32)], ids=str)
def test_step_refuses_another_cache(calls, cache):
    with pytest.raises(ValueError, match="cache"):
        _model(cache=cache).step(torch.zeros(CHUNK), torch.zeros(COND, dtype=torch.bfloat16), 0)
    assert not calls
