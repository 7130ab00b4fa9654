"""The forward's blocks hold one query stream each where the chip has an SM for every stream (up to 148), and two where it has
not (two heads, or two tiles where the group size is odd): a sequence has the same result in either kind of call, bit for
bit, and the one it has in a packed sample."""
import pytest
import torch

import paper_2509_15763_b200 as ug

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# raw tokens, ratio, window, query heads, KV heads, head_dim, sinks, sequences in the large call
SHAPES = [(448, 7, 64, 1, 1, 64, 0, 60),       # odd group, 5 tiles a head: 5 blocks of one stream; tile pairs
          (448, 7, 64, 3, 1, 128, 0, 30),
          (35 * 128, 128, 300, 4, 2, 128, 0, 2),  # 144 streams, and 288
          (36 * 128 - 128, 64, 300, 4, 4, 64, 3, 2),  # 148, and 296
          (130, 13, 26, 8, 2, 128, 130, 12),   # sinks of two tiles, ragged ends
          (1, 1, 0, 2, 1, 64, 0, 90)]


def _fwd(p, q, k, v):
    o = torch.full_like(q, float("nan"))
    lse = torch.full((p.batch, p.num_q_heads, q.shape[1]), float("nan"), device=DEV)
    ug.unigist_attn_fwd(p, q, k, v, o, lse)
    ug.unigist_device_status()
    return o, lse


@pytest.mark.parametrize("raw,ratio,window,hq,hkv,dim,sinks,many", SHAPES)
def test_alone_and_in_a_batch(raw, ratio, window, hq, hkv, dim, sinks, many):
    one, all_ = (ug.Problem(b, raw, ratio, window, hq, hkv, dim, num_sinks=sinks) for b in (1, many))
    n = ug.unigist_total_len(one)
    tiles = sum(-(-x // 128) for x in (sinks, raw, raw // ratio))
    assert tiles * hq <= 148 < tiles * hq * many
    g = torch.Generator(device=DEV).manual_seed(raw + hq)
    q, k, v = (torch.randn(many, n, h, dim, generator=g, device=DEV).bfloat16() for h in (hq, hkv, hkv))
    o, lse = _fwd(all_, q, k, v)
    assert not torch.isnan(o).any() and not torch.isnan(lse).any()
    for b in (0, many // 2, many - 1):
        o1, lse1 = _fwd(one, q[b:b + 1].contiguous(), k[b:b + 1].contiguous(), v[b:b + 1].contiguous())
        assert torch.equal(o1[0], o[b]) and torch.equal(lse1[0], lse[b])
    # as a packed sample of two documents (its streams together decide), each as it is alone
    flat = [x[:2].reshape(1, 2 * n, x.shape[2], dim) for x in (q, k, v)]
    o2, lse2 = torch.empty_like(flat[0]), torch.empty(2 * n * hq, device=DEV)
    ug.unigist_attn_fwd_docs(one, [raw, raw], *flat, o2, lse2)
    ug.unigist_device_status()
    assert torch.equal(o2.reshape(2, n, hq, dim), o[:2]) and torch.equal(lse2.reshape(2, hq, n), lse[:2])
