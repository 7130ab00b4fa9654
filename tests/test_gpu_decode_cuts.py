"""Every way a decode call is cut, against the oracle: clusters of 1 to 16 blocks per (sequence, KV head), the flat walk
over all sequences' pages (fewer pages than shares, sequences inside one share, cut once and cut many times, empty
ones between them), and the least scratch that is accepted."""
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
]


@pytest.mark.parametrize("least", [False, True])
@pytest.mark.parametrize("Hq,Hkv,lens,width", CASES)
def test_decode_cuts(Hq, Hkv, lens, width, least):
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
    size = ug.unigist_decode_workspace_bytes(S, Hq, Hkv, D, width)
    if least:  # what one partial result per sequence and query head takes, or as much more as the call insists on
        size = -(-S * Hq * (D + 2) * 4 // 256) * 256
    ws = torch.empty(size, dtype=torch.uint8, device=DEV)
    o = torch.full((S, Hq, D), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((S, Hq), float("nan"), dtype=torch.float32, device=DEV)
    args = [x.to(DEV) for x in (q, kc, vc, table, torch.tensor(lens, dtype=torch.int32))]
    try:
        ug.unigist_decode(*args, o, lse, ws)
    except ug.UnigistError as e:
        assert least and e.code == 4  # UNIGIST_ERR_WORKSPACE
        need = int(str(e).split("decode needs ")[1].split()[0])
        assert need <= ug.unigist_decode_workspace_bytes(S, Hq, Hkv, D, width)
        ug.unigist_decode(*args, o, lse, torch.empty(need, dtype=torch.uint8, device=DEV))
    torch.cuda.synchronize()
    ug.unigist_device_status()
    for i, n in enumerate(lens):
        if n == 0:
            assert (o[i] == 0).all() and (lse[i] == -np.inf).all()
            continue
        kl, vl = (f64(c[table[i, :used[i]].long()].permute(0, 2, 1, 3).reshape(-1, Hkv, D)[:n]) for c in (kc, vc))
        oo, ll = oracle.decode(D ** -0.5, f64(q[i:i + 1]), [kl], [vl])
        check_close(f"O of sequence {i}", f64(o[i:i + 1]), oo, TOL_O_MAX, TOL_O_MEAN)
        check_close(f"LSE of sequence {i}", f64(lse[i:i + 1]), ll, TOL_LSE)
