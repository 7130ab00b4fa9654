"""Kernels that run beside the one before them (the dQ kernel of the two-kernel backward beside dK / dV): the same bits as with
a synchronisation after every call, whatever follows at once and whatever the workspace held before; dQ in place of Q or dO."""
import pytest
import torch

import paper_2509_15763_b200 as ug

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _problem(batch, raw, ratio, window, hq, hkv, dim, sinks):
    return ug.Problem(batch, raw, ratio, window, hq, hkv, dim, num_sinks=sinks, flags=ug.FLAG_DETERMINISTIC_DQ if dim == 128 else 0)


def _inputs(p, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = ug.unigist_total_len(p)

    def t(h):
        return torch.randn(p.batch, n, h, p.head_dim, generator=g, device=DEV).bfloat16()

    x = {"q": t(p.num_q_heads), "k": t(p.num_kv_heads), "v": t(p.num_kv_heads), "do": t(p.num_q_heads)}
    x["o"], x["lse"] = torch.empty_like(x["q"]), torch.empty(p.batch, p.num_q_heads, n, device=DEV)
    ug.unigist_attn_fwd(p, x["q"], x["k"], x["v"], x["o"], x["lse"])
    return x


def _bwd(p, x, ws, dq, dk, dv):
    ug.unigist_attn_bwd(p, x["q"], x["k"], x["v"], x["o"], x["lse"], x["do"], dq, dk, dv, ws)


SHAPES = [(1, 6, 3, 4, 1, 1, 64, 0), (1, 448, 7, 64, 1, 1, 64, 0), (2, 1400, 7, 300, 8, 2, 64, 5), (3, 96, 4, 50, 12, 1, 64, 3),
          (1, 640, 5, 128, 8, 2, 128, 130)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_backward_back_to_back(shape):
    p = _problem(*shape)
    ws = torch.empty(ug.unigist_workspace_bytes(p, ug.OP_BWD), dtype=torch.uint8, device=DEV)
    xs = [_inputs(p, s) for s in (1, 2)]

    def buffers(x):  # the gradients, and their unshifted copies
        return [torch.full_like(x[n], float("nan")) for n in ("q", "k", "v") * 2]

    want = [buffers(x) for x in xs]
    for x, w in zip(xs, want):
        torch.cuda.synchronize()
        _bwd(p, x, ws, *w[:3])
        torch.cuda.synchronize()
        for a, b in zip(w[:3], w[3:]):
            ug.unigist_gist_unshift(p, a, b)
    for _ in range(3):  # the two inputs in turn through one workspace, each gradient read by the next kernel at once
        got = [buffers(x) for x in xs]
        torch.cuda.synchronize()
        for x, g in zip(xs, got):
            _bwd(p, x, ws, *g[:3])
            for a, b in zip(g[:3], g[3:]):
                ug.unigist_gist_unshift(p, a, b)
        ug.unigist_device_status()
        for g, w in zip(got, want):
            assert all(torch.equal(a, b) for a, b in zip(g, w))


@pytest.mark.parametrize("over", ["q", "do"])
@pytest.mark.parametrize("shape", SHAPES[2:], ids=str)
def test_dq_in_place(shape, over):
    p = _problem(*shape)
    ws = torch.empty(ug.unigist_workspace_bytes(p, ug.OP_BWD), dtype=torch.uint8, device=DEV)
    x = _inputs(p, 3)
    want = [torch.empty_like(x[n]) for n in ("q", "k", "v")]
    _bwd(p, x, ws, *want)
    got = [x[over], torch.empty_like(x["k"]), torch.empty_like(x["v"])]
    _bwd(p, x, ws, *got)
    ug.unigist_device_status()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
