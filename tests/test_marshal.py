"""What the binding's marshalling refuses before any C call (no GPU needed)."""
import subprocess
import sys
from pathlib import Path

import numpy as np
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


def test_a_problem_of_numpy_integers_is_a_problem():
    fields = [np.int64(1), np.int32(16), np.int16(4), np.uint8(4), np.int64(1), np.int64(1), np.int64(64)]
    p = ug.Problem(*fields, num_sinks=np.int64(0), flags=np.uint32(0))
    assert ug.unigist_total_len(p) == 20  # the size queries take it
    with pytest.raises(ValueError, match="contiguous CUDA tensors"):  # ... and so do the calls: on to their tensors
        ug.unigist_gist_shift(p, t(), t())
    with pytest.raises(TypeError):
        ug.unigist_gist_shift(ug.Problem(np.float32(1), *fields[1:]), t(), t())


# One call of every enqueueing function with a fake CUDA tensor `x` as one of its tensors: inside a transform x has no storage,
# so its address cannot be taken.
NO_STORAGE = """
import sys, types
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
import paper_2509_15763_b200 as ug

P, st = ug.Problem(1, 16, 4, 4, 1, 1, 64), types.SimpleNamespace(cuda_stream=0)
calls = [
    lambda x, t: ug.unigist_gist_shift(P, x, t, stream=st),
    lambda x, t: ug.unigist_gist_unshift(P, t, x, stream=st),
    lambda x, t: ug.unigist_rope(P, t, x, 1e4, stream=st),
    lambda x, t: ug.unigist_attn_fwd(P, t, t, x, t, t, stream=st),
    lambda x, t: ug.unigist_attn_bwd(P, *[t] * 9, x, stream=st),
    lambda x, t: ug.unigist_attn_fwd_docs(P, [16], x, t, t, t, t, stream=st),
    lambda x, t: ug.unigist_attn_bwd_docs(P, [16], *[t] * 5, x, t, t, t, t, stream=st),
    lambda x, t: ug.unigist_kv_compact(P, t, x, t, t, t, t, stream=st),
    lambda x, t: ug.unigist_prefill_chunk(P, 0, 1, *[t] * 9, x, stream=st),
    lambda x, t: ug.unigist_cache_state_init(P, 0, x, stream=st),
    lambda x, t: ug.unigist_cache_append(P, x, t, False, *[t] * 5, stream=st),
    lambda x, t: ug.unigist_decode_step(P, x, *[t] * 8, stream=st),
    lambda x, t: ug.unigist_decode(x[0], *[t] * 7, stream=st),
    lambda x, t: ug.unigist_decode_static(x[0], *[t] * 6, stream=st),
]
before = ug.unigist_launch_count()
with FakeTensorMode():
    t = torch.zeros(1, 20, 1, 64, dtype=torch.bfloat16, device="cuda")
    for call in calls:
        def f(x):
            call(x, t)
            return x.float().sum()
        for run in (lambda: torch.func.vmap(f)(torch.stack([t, t])), lambda: torch.func.grad(f)(t),
                    lambda: torch.func.jvp(f, (t,), (t,))):
            try:
                run()
            except RuntimeError as e:
                assert "Cannot access data pointer" in str(e), e
            else:
                raise AssertionError("accepted")
assert ug.unigist_launch_count() == before
print("refused", 3 * len(calls))
"""


def test_tensors_without_storage_are_refused():
    run = subprocess.run([sys.executable, "-c", NO_STORAGE], cwd=Path(__file__).resolve().parent.parent, capture_output=True, text=True)
    assert run.returncode == 0 and "refused 42" in run.stdout, run.stderr[-2000:]
