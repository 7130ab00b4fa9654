"""What the binding's marshalling refuses before any C call (no GPU needed)."""
import pytest
import torch

import paper_2509_15763_b200 as ug

P = ug.Problem(1, 16, 4, 4, 1, 1, 64)


def t():
    return torch.zeros(1, 20, 1, 64, dtype=torch.bfloat16)


@pytest.mark.parametrize("call", [
    lambda: ug.unigist_gist_shift(P, t(), t()),
    lambda: ug.unigist_rope(P, t(), t(), 10000.0),
    lambda: ug.unigist_attn_fwd(P, t(), t(), t(), t(), t()),
    lambda: ug.unigist_attn_bwd(P, *[t()] * 10),
    lambda: ug.unigist_attn_fwd_docs(P, [16], t(), t(), t(), t(), t()),
    lambda: ug.unigist_kv_compact(P, t(), t(), t(), t(), t(), t()),
    lambda: ug.unigist_prefill_chunk(P, 0, 1, *[t()] * 10),
    lambda: ug.unigist_cache_state_init(P, 0, t()),
    lambda: ug.unigist_cache_append(P, t(), t(), False, *[t()] * 5),
    lambda: ug.unigist_decode_step(P, *[t()] * 8),
    lambda: ug.unigist_decode(*[t()] * 6),
    lambda: ug.unigist_decode_static(*[t()] * 6),
])
def test_host_tensors_are_refused(call):
    before = ug.unigist_launch_count()
    with pytest.raises(ValueError, match="contiguous CUDA tensors"):
        call()
    assert ug.unigist_launch_count() == before


def test_wrong_kinds_of_arguments_are_refused():
    with pytest.raises(TypeError):
        ug.unigist_gist_shift(P, [1, 2], t())
    with pytest.raises(TypeError):
        ug.unigist_gist_shift(ug.Problem(1.5, 16, 4, 4, 1, 1, 64), t(), t())
    with pytest.raises(AttributeError):
        ug.unigist_gist_shift(object(), t(), t())
    with pytest.raises((TypeError, ValueError)):
        ug.unigist_attn_fwd_docs(P, ["x"], *[t()] * 5)
    with pytest.raises(TypeError):
        ug.unigist_attn_fwd_docs(P, 16, *[t()] * 5)
