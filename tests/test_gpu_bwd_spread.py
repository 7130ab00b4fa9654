"""The fused backward where the longest sink or gist walk is cut to spread it over idle SMs: against the oracle, shifted and
interleaved, dK and dV the same bits twice; and with a workspace that has no room for the partial sums."""
import numpy as np
import pytest
import torch

import paper_2509_15763_b200 as ug
from paper_2509_15763_b200 import synth
from oracle import oracle

from gpu_util import TOL_GRAD, check_close, f64, problem_of, run_attention, run_attention_interleaved

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [
    synth.Workload("one_gist_tile", 1, 1024, 8, 64, 8, 1, 128, seed=601),            # 9 tiles in chunks of 3 - 4
    synth.Workload("sinks_two_tiles", 1, 896, 16, 64, 8, 1, 128, num_sinks=130, seed=602),
    synth.Workload("ragged_batch", 2, 128 * 6 + 8, 8, 40, 8, 2, 128, num_sinks=1, seed=603),
]


def _base_bytes(w):
    al, tokens = (lambda x: -(-x // 256) * 256), w.batch * ug.unigist_total_len(problem_of(w))
    return al(tokens * w.num_q_heads * 4) + al(tokens * w.num_q_heads * 128 * 4)


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
@pytest.mark.parametrize("run", [run_attention, run_attention_interleaved], ids=["shifted", "interleaved"])
def test_cut_walks(w, run):
    assert ug.unigist_workspace_bytes(problem_of(w), ug.OP_BWD) > _base_bytes(w)  # partial sums: some walk is cut
    out, again = run(w), run(w)
    k, scale, inp = oracle.window_units(w.window, w.ratio), w.head_dim ** -0.5, out["inputs"]
    want = oracle.attn_bwd(w.num_sinks, w.raw_len, w.ratio, k, scale, *(f64(inp[n]) for n in ("q", "k", "v", "dout")))
    for name, ref in zip(("dq", "dk", "dv"), want):
        check_close(name, f64(out[name]), np.asarray(ref), TOL_GRAD)
    assert torch.equal(out["dk"], again["dk"]) and torch.equal(out["dv"], again["dv"])


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_without_room_for_partial_sums(w):
    p, n = problem_of(w), ug.unigist_total_len(problem_of(w))
    g = torch.Generator(device=DEV).manual_seed(w.seed)
    q, k, v, do = (torch.randn(w.batch, n, h, 128, generator=g, device=DEV).bfloat16()
                   for h in (w.num_q_heads, w.num_kv_heads, w.num_kv_heads, w.num_q_heads))
    o, lse = torch.empty_like(q), torch.empty(w.batch, w.num_q_heads, n, device=DEV)
    ug.unigist_attn_fwd(p, q, k, v, o, lse)

    def bwd(size):
        # the bytes behind the size that is given are not the call's
        ws = torch.full((size + 4096,), 7, dtype=torch.uint8, device=DEV)
        grads = [torch.full_like(x, float("nan")) for x in (q, k, v)]
        ug.unigist_attn_bwd(p, q, k, v, o, lse, do, *grads, ws[:size])
        ug.unigist_device_status()
        assert bool((ws[size:] == 7).all())
        return grads

    full, least = ug.unigist_workspace_bytes(p, ug.OP_BWD), _base_bytes(w)
    cut, uncut, between = bwd(full), bwd(least), bwd(full - 16)
    for a, b in zip(cut, uncut):  # two roundings of one fp32 sum to bf16 (dQ, a few: its sums have no fixed order)
        assert float((a.float() - b.float()).norm()) <= 2 ** -8 * float(b.float().norm())
    assert torch.equal(uncut[1], between[1]) and torch.equal(uncut[2], between[2])
    with pytest.raises(ug.UnigistError):
        bwd(least - 16)


@pytest.mark.parametrize("docs", [[1024, 64], [32, 1200, 1200, 8]], ids=str)
def test_packed_sample(docs):
    p = ug.Problem(1, 8, 8, 64, 8, 1, 128, num_sinks=2)
    n = ug.unigist_docs_total_len(p, docs)
    g = torch.Generator(device=DEV).manual_seed(610 + len(docs))
    q, k, v, do = (torch.randn(1, n, h, 128, generator=g, device=DEV).bfloat16() for h in (8, 1, 1, 8))
    o, lse = torch.empty_like(q), torch.empty(8 * n, device=DEV)
    ug.unigist_attn_fwd_docs(p, docs, q, k, v, o, lse)
    al = lambda x: -(-x // 256) * 256
    full, least = ug.unigist_docs_workspace_bytes(p, ug.OP_BWD, docs), al(n * 8 * 4) + al(n * 8 * 128 * 4)
    assert full > least
    got = []
    for size in (full, full, least):
        ws = torch.full((size + 4096,), 7, dtype=torch.uint8, device=DEV)
        got.append([torch.full_like(x, float("nan")) for x in (q, k, v)])
        ug.unigist_attn_bwd_docs(p, docs, q, k, v, o, lse, do, *got[-1], ws[:size])
        ug.unigist_device_status()
        assert bool((ws[size:] == 7).all())
    assert torch.equal(got[0][1], got[1][1]) and torch.equal(got[0][2], got[1][2])
    for a, b in zip(got[0], got[2]):
        assert float((a.float() - b.float()).norm()) <= 2 ** -8 * float(b.float().norm())
    with pytest.raises(ug.UnigistError):
        ug.unigist_attn_bwd_docs(p, docs, q, k, v, o, lse, do, *got[0], ws[:least - 16])


@pytest.mark.parametrize("sinks", [0, 130])
def test_packed_sample_with_several_cut_documents(sinks):
    """The partial sums of all units that are cut (runs of several sequences and several KV heads among them) are added by one
    kernel: at most four launches in all, and eight where a sample has more than twelve units."""
    p, ratio = ug.Problem(1, 8, 8, 64, 16, 2, 128, num_sinks=sinks), 8
    for docs, launches in (([1200, 1200, 1024, 64, 904], 4), ([1200 - ratio * i for i in range(12)] + [1600, 8], 8)):
        n = ug.unigist_docs_total_len(p, docs)
        g = torch.Generator(device=DEV).manual_seed(620 + len(docs) + sinks)
        q, k, v, do = (torch.randn(1, n, h, 128, generator=g, device=DEV).bfloat16() for h in (16, 2, 2, 16))
        o, lse = torch.empty_like(q), torch.empty(16 * n, device=DEV)
        ug.unigist_attn_fwd_docs(p, docs, q, k, v, o, lse)
        al = lambda x: -(-x // 256) * 256
        full, least = ug.unigist_docs_workspace_bytes(p, ug.OP_BWD, docs), al(n * 16 * 4) + al(n * 16 * 128 * 4)
        assert full > least
        got = []
        for size in (full, least):
            ws = torch.full((size + 4096,), 7, dtype=torch.uint8, device=DEV)
            got.append([torch.full_like(x, float("nan")) for x in (q, k, v)])
            before = ug.unigist_launch_count()
            ug.unigist_attn_bwd_docs(p, docs, q, k, v, o, lse, do, *got[-1], ws[:size])
            assert ug.unigist_launch_count() - before <= launches
            ug.unigist_device_status()
            assert bool((ws[size:] == 7).all())
        for a, b in zip(*got):
            assert float((a.float() - b.float()).norm()) <= 2 ** -8 * float(b.float().norm())
