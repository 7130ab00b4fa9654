"""Every way a decode call is cut, against the oracle: clusters of 1 to 16 blocks per (sequence, KV head), the even split
with a second kernel, the flat walk over all sequences' pages (fewer pages than shares, sequences inside one share, cut once
and cut many times, empty ones between them, more sequences than a block has threads), and every size of scratch from the
least that is accepted."""
import numpy as np
import pytest
import torch

import paper_2509_15763_b200 as ug
from oracle import oracle
from gpu_util import TOL_LSE, TOL_O_MAX, TOL_O_MEAN, check_close, f64

pytestmark = pytest.mark.gpu
PG = ug.PAGE_TOKENS
DEV = "cuda:0"

# (Hq, Hkv, lengths, width of the block table in pages)
CASES = [
    (8, 2, [130], 3),                            # one round of a block's three warps: no cluster
    (8, 2, [1], 9), (8, 1, [64 * 9], 9),         # clusters; some of their blocks have no page
    (4, 4, [64 * 40 + 1, 700], 41),
    (16, 2, [64 * 90], 90),                      # clusters of 16
    (8, 2, [100, 0, 65], 700),                   # flat: fewer pages than shares, an empty sequence
    (8, 1, [64 * 30, 0, 0, 64, 1, 64 * 61 + 3], 700),
    (6, 2, [17 * (i % 13) for i in range(50)], 160),                    # flat: several sequences inside one share
    (8, 8, [3000, 1, 2999, 64, 63, 65, 0, 1500] * 5, 47),               # 40 sequences, 320 pairs
    (4, 4, [40 + 3 * i for i in range(80)], 7),                         # many short walks: one block each
    (1, 1, [(37 * i) % 300 for i in range(300)], 20),                   # three sequences per thread in the page counts
    (1, 1, [(37 * i) % 300 for i in range(384)], 20),                   # ... with the runs ending at the last sequence
    (1, 1, [(37 * i) % 300 for i in range(769)], 20),                   # seven, the last threads without any
    (2, 1, [5000] + [(29 * i) % 150 for i in range(1099)] + [64 * 70], 90),  # long sequences among short ones
    (64, 8, [40 + 7 * (i % 30) for i in range(230)], 80),               # more than 8 MiB of scratch asked for
    (8, 1, [64 * 192], 192), (8, 2, [6400, 0], 100), (32, 8, [64 * 99 + 5], 144),  # few pairs: the even split
    (8, 1, [0], 192), (8, 1, [1], 192),                                 # ... of nothing, of one page
    (32, 8, [64 * 79 + 1, 3], 80),                                      # more clusters of 16 than fit
    (160, 160, [900, 17], 40),                                          # more KV heads than SMs
]


def _inputs(Hq, Hkv, lens, width):
    S, D = len(lens), 128
    g = torch.Generator().manual_seed(S * 1000 + width)
    used = [-(-n // PG) for n in lens]
    blocks = sum(used) + 1
    kc, vc = (torch.randn(blocks, Hkv, PG, D, generator=g).to(torch.bfloat16) for _ in range(2))
    order = torch.randperm(sum(used), generator=g).to(torch.int32)
    table = torch.full((S, width), blocks - 1, dtype=torch.int32)
    at = 0
    for i, n in enumerate(used):
        table[i, :n] = order[at:at + n]
        at += n
    q = torch.randn(S, Hq, D, generator=g).to(torch.bfloat16)
    return q, kc, vc, table, torch.tensor(lens, dtype=torch.int32)


def _check(inputs, o, lse):
    q, kc, vc, table, lens = inputs
    Hkv, D = kc.shape[1], 128
    for i, n in enumerate(lens.tolist()):
        if n == 0:
            assert (o[i] == 0).all() and (lse[i] == -np.inf).all()
            continue
        kl, vl = (f64(c[table[i, :-(-n // PG)].long()].permute(0, 2, 1, 3).reshape(-1, Hkv, D)[:n]) for c in (kc, vc))
        oo, ll = oracle.decode(D ** -0.5, f64(q[i:i + 1]), [kl], [vl])
        check_close(f"O of sequence {i}", f64(o[i:i + 1]), oo, TOL_O_MAX, TOL_O_MEAN)
        check_close(f"LSE of sequence {i}", f64(lse[i:i + 1]), ll, TOL_LSE)


@pytest.mark.parametrize("least", [False, True])
@pytest.mark.parametrize("Hq,Hkv,lens,width", CASES)
def test_decode_cuts(Hq, Hkv, lens, width, least):
    S, D = len(lens), 128
    inputs = _inputs(Hq, Hkv, lens, width)
    size = ug.unigist_decode_workspace_bytes(S, Hq, Hkv, D, width)
    if least:  # what one partial result per sequence and query head takes, or as much more as the call insists on
        size = -(-S * Hq * (D + 2) * 4 // 256) * 256
    ws = torch.empty(size, dtype=torch.uint8, device=DEV)
    o = torch.full((S, Hq, D), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((S, Hq), float("nan"), dtype=torch.float32, device=DEV)
    args = [x.to(DEV) for x in inputs]
    try:
        ug.unigist_decode(*args, o, lse, ws)
    except ug.UnigistError as e:
        assert least and e.code == 4  # UNIGIST_ERR_WORKSPACE
        need = int(str(e).split("decode needs ")[1].split()[0])
        assert need <= ug.unigist_decode_workspace_bytes(S, Hq, Hkv, D, width)
        ug.unigist_decode(*args, o, lse, torch.empty(need, dtype=torch.uint8, device=DEV))
    torch.cuda.synchronize()
    ug.unigist_device_status()
    _check(inputs, o, lse)
    if not least and size <= ug.DECODE_STATIC_SCRATCH_BYTES:  # the same cut, bit for bit, with the built-in scratch
        o2, lse2 = torch.full_like(o, float("nan")), torch.full_like(lse, float("nan"))
        ug.unigist_decode_static(*args, o2, lse2)
        assert torch.equal(o, o2) and torch.equal(lse, lse2)


@pytest.mark.parametrize("Hq,Hkv,lens,width", [(32, 8, [64 * 3 * (i % 5) + 1 for i in range(37)], 144),  # one part each suffices
                                               (8, 1, [64 * 20 + i for i in range(5)], 300),
                                               (8, 8, [700] * 40, 47)])
def test_every_size_of_scratch(Hq, Hkv, lens, width):
    """From the least that is accepted to more than is asked for, in steps that do not divide the parts."""
    S, D = len(lens), 128
    inputs = _inputs(Hq, Hkv, lens, width)
    args = [x.to(DEV) for x in inputs]
    o = torch.empty(S, Hq, D, dtype=torch.bfloat16, device=DEV)
    lse = torch.empty(S, Hq, dtype=torch.float32, device=DEV)
    with pytest.raises(ug.UnigistError) as e:
        ug.unigist_decode(*args, o, lse, torch.empty(256, dtype=torch.uint8, device=DEV))
    least = int(str(e.value).split("decode needs ")[1].split()[0])
    ideal = ug.unigist_decode_workspace_bytes(S, Hq, Hkv, D, width)
    assert least <= ideal
    guard = 4096
    for size in sorted({least, least + 16, 655360, (least + ideal) // 2 // 16 * 16, ideal - 16, ideal, ideal + 100000}):
        if size < least:
            continue
        buf = torch.full((size + guard,), 0xA5, dtype=torch.uint8, device=DEV)
        o.fill_(float("nan"))
        lse.fill_(float("nan"))
        ug.unigist_decode(*args, o, lse, buf[:size])
        torch.cuda.synchronize()
        assert (buf[size:] == 0xA5).all()  # nothing behind the workspace
        _check(inputs, o, lse)


@pytest.mark.parametrize("width", [3, 9, 100, 700])  # one block, a cluster, the even split, the flat walk
@pytest.mark.parametrize("n", [1, 130])
def test_infinities_in_v(width, n):
    """A visible infinity in V comes out as that infinity (both signs in one column: NaN), whatever the rounding of its
    weight; the other columns are as exact as ever."""
    Hq, Hkv, D = 8, 2, 128
    g = torch.Generator().manual_seed(n + width)
    pages = -(-n // PG)
    kc, vc = (torch.randn(pages, Hkv, PG, D, generator=g).to(torch.bfloat16) for _ in range(2))
    inf = float("inf")
    for i, column in enumerate((0, 9, 77)):  # the token that holds an infinity: the first one, and where there are more, others
        t = (0, n // 2, n - 1)[i]
        vc[t // PG, :, t % PG, column] = inf if i % 2 == 0 else -inf
    if n > 1:
        vc[0, :, 0, 127], vc[0, :, 1, 127] = inf, -inf
    q = (0.5 * torch.randn(1, Hq, D, generator=g)).to(torch.bfloat16)  # (every weight stays above zero)
    table = torch.zeros(1, width, dtype=torch.int32)
    table[0, :pages] = torch.arange(pages)
    ws = torch.empty(ug.unigist_decode_workspace_bytes(1, Hq, Hkv, D, width), dtype=torch.uint8, device=DEV)
    o = torch.zeros(1, Hq, D, dtype=torch.bfloat16, device=DEV)
    ug.unigist_decode(*(x.to(DEV) for x in (q, kc, vc, table, torch.tensor([n], dtype=torch.int32))), o, None, ws)
    torch.cuda.synchronize()
    got = f64(o[0])
    assert (got[:, 0] == inf).all() and (got[:, 9] == -inf).all() and (got[:, 77] == inf).all()
    assert n == 1 or np.isnan(got[:, 127]).all()
    rest = [c for c in range(D) if c not in (0, 9, 77, 127)]
    kl, vl = (f64(c.permute(0, 2, 1, 3).reshape(-1, Hkv, D)[:n]) for c in (kc, vc))
    want = oracle.decode(D ** -0.5, f64(q), [kl], [np.where(np.isfinite(vl), vl, 0.0)])[0][0]
    check_close("the other columns", got[:, rest], want[:, rest], TOL_O_MAX, TOL_O_MEAN)
