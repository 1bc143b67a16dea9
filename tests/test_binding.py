"""Argument checks of the extension module, on tensors without memory (fake CUDA tensors): nothing is launched, and a call
that passes every check ends where the current stream is asked for."""
import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

from paper_2505_20776_b200 import api

NO_ENTRY = 0
NO_POINTER = "data pointer"


def _fake(*shape, dtype=torch.float32):
    with FakeTensorMode(allow_non_fake_inputs=True):
        return torch.empty(*shape, dtype=dtype, device="cuda")


def _attn(name, ws):
    q, kv = _fake(2, 4, 64, dtype=torch.bfloat16), _fake(2, 2, 64, dtype=torch.bfloat16)
    i, f = _fake(2, dtype=torch.int32), _fake(8)
    call = getattr(api._binding(), name)
    if name == "verify_attn":
        return call(NO_ENTRY, api.AttnDesc(), q, kv, kv, kv, kv, i, q, f, None, ws, i)
    return call(NO_ENTRY, api.AttnDesc(), q, kv, kv, i, kv, kv, i, q, f, ws, i)


def _select_gather(out, k=2, C=1, draft=None):
    i = _fake(8, dtype=torch.int32)
    draft = _fake(1, 100, 4, 8, dtype=torch.bfloat16) if draft is None else draft
    return api._binding().select_gather(NO_ENTRY, _fake(1, 4), 1, 4, 0, 100, C, k, 0, 0, draft, draft, i, i, out, out, i, i)


@pytest.mark.parametrize("call", [lambda t: _attn("verify_attn", t), lambda t: _attn("draft_attn", t), _select_gather])
def test_a_tensor_without_memory_raises_before_the_lock_is_released(call):
    """A workspace or an output inside vmap has no data pointer: an ordinary error, raised while the interpreter lock is held."""
    batched = _fake(1, 4096, dtype=torch.bfloat16)
    with pytest.raises(RuntimeError, match=NO_POINTER):
        torch.func.vmap(lambda t: call(t))(batched)


@pytest.mark.parametrize("k,C,layers,heads,dim", [
    (2 ** 31 - 1, 2 ** 31 - 1, 1, 4, 8),           # the product wraps to a negative number
    (2 ** 14, 2 ** 14, 2 ** 15, 2 ** 11, 2 ** 10), # to zero, with every factor in the library's range
    (9, 1, 1, 4, 8),                               # one token too many
])
def test_select_gather_output_size_does_not_wrap(k, C, layers, heads, dim):
    """A compact cache that is too small for [layers][k * C][heads][dim] is refused whatever the product."""
    draft = _fake(1, 1, heads, dim, dtype=torch.bfloat16).expand(layers, 100, heads, dim)
    with pytest.raises(ValueError, match="must be contiguous and hold"):
        _select_gather(_fake(8 * 32, dtype=torch.bfloat16), k, C, draft)
