"""The native marshalling takes and refuses what the Python binding in front of the C ABI did (no GPU: every call ends in a refusal)."""
import types

import pytest
import torch

from paper_2607_14695_b200 import binding as rb
from paper_2607_14695_b200 import build as rbuild

NO_CACHE = types.SimpleNamespace(handle=None)


@pytest.fixture(scope="module", autouse=True)
def built():
    rbuild.build()


def _refused(call, *args, **kw):
    with pytest.raises(rb.ReflexError) as e:
        call(*args, stream=0, **kw)
    return e.value.code


def test_stacked_gate_weights_are_no_single_layer():
    x, cond, b = torch.zeros(1, 1, 64), torch.zeros(1, 8), torch.zeros(8)
    with pytest.raises(ValueError):
        rb.reflex_adarmsnorm(x, torch.zeros_like(x), cond, torch.zeros(8, 8, 8), b, torch.zeros(64, 8), b, stream=0)


@pytest.mark.parametrize("call", [rb.reflex_cache_init_static, rb.reflex_cache_stage_static])
def test_prefix_lengths(call):
    k = torch.zeros(2, 1, 4, 1, 32)
    # as many as streams, or more (the first ones count), reach the library
    assert _refused(call, NO_CACHE, [0, 1], k, k, S=[4, 4]) == _refused(call, NO_CACHE, [0, 1], k, k, S=[4, 4, 1]) == rb.ERR_INVALID_ARG
    with pytest.raises(ValueError):
        call(NO_CACHE, [0, 1], k, k, S=[4], stream=0)


@pytest.mark.parametrize("eps", [1e-6, "1e-6", torch.tensor(1e-6), True, -1.0])
def test_numbers_of_any_kind(eps):
    x = torch.zeros(1, 1, 64)
    gate = torch.zeros(1, 64)
    bad_width = _refused(rb.reflex_adarmsnorm, x[..., :12].contiguous(), x[..., :12].contiguous(), None, None, None, None, None, gate_buf=gate, eps=eps)
    assert bad_width == rb.ERR_SHAPE
