"""A thread whose first CUDA call is a call of this library (a server's worker thread): tensor maps need a current context."""
import threading

import pytest
import torch

import paper_2509_15763_b200 as ug

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def bf16(*shape):
    return torch.randn(*shape, device=DEV, generator=torch.Generator(DEV).manual_seed(5)).to(torch.bfloat16)


def decode():
    q, kc, vc = bf16(2, 8, 128), bf16(6, 2, 64, 128), bf16(6, 2, 64, 128)
    table = torch.arange(6, dtype=torch.int32, device=DEV).reshape(2, 3)
    lens = torch.tensor([150, 70], dtype=torch.int32, device=DEV)
    o, lse = torch.zeros_like(q), torch.zeros(2, 8, device=DEV)
    ws = torch.empty(ug.unigist_decode_workspace_bytes(2, 8, 2, 128, 3), dtype=torch.uint8, device=DEV)
    return (o, lse), lambda stream: ug.unigist_decode(q, kc, vc, table, lens, o, lse, ws, stream=stream)


def forward():
    p = ug.Problem(1, 256, 8, 64, 4, 2, 128)
    n = ug.unigist_total_len(p)
    q, k, v = bf16(1, n, 4, 128), bf16(1, n, 2, 128), bf16(1, n, 2, 128)
    o, lse = torch.zeros_like(q), torch.zeros(1, 4, n, device=DEV)
    return (o, lse), lambda stream: ug.unigist_attn_fwd(p, q, k, v, o, lse, stream=stream)


@pytest.mark.parametrize("make", [decode, forward])
def test_first_cuda_call_of_a_thread(make):
    out, call = make()
    stream = torch.cuda.current_stream()
    call(stream)
    torch.cuda.synchronize()
    want = [x.clone() for x in out]
    for x in out:
        x.zero_()
    torch.cuda.synchronize()
    failed = []

    def work():
        try:
            call(stream)
        except Exception as e:  # noqa: BLE001 - handed to the test's thread
            failed.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    assert all(torch.equal(a, b) for a, b in zip(out, want))
