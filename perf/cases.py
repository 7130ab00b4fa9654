"""Workloads of the library's public calls, with the work each cannot do without and how close two correct
implementations come to each other.

A case is one of six things a program does with this library; `kind` says which:

  train    one attention layer, forward and backward.  `tensors` says how the tensors are ordered: "interleaved"
           (the gist shift happens in the tile addressing), "shifted" (explicit gist shift of q, k, v, dO before and
           unshift of o, dq, dk, dv after) or "rope" (rotary embedding of q and k fused with the shift, its transpose
           fused with the unshift of dq and dk)
  packed   a packed training sample under cross-document masking, forward and backward
  prefill  forward over a whole prompt, then compaction of its keys and values into the paged cache
  chunks   the same prompt fed chunk by chunk over the compressed cache
  decode   one query per sequence over the paged compressed cache
  loop     token-by-token generation of two gist units: every token is appended to the cache and attends to it (the
           first token of the second unit evicts the unit that has left the window)
"""
import math

import torch

import paper_2509_15763_b200 as ug

PAGE = ug.PAGE_TOKENS
DEV = "cuda:0"
ROPE_BASE = 500000.0


def _train(name, batch, raw_len, ratio, window, hq, hkv, dim, sinks=0, tensors="interleaved", dout_fp32=False,
           fixed_dq=False):
    return {"name": name, "kind": "train", "batch": batch, "raw_len": raw_len, "ratio": ratio, "window": window, "hq": hq,
            "hkv": hkv, "dim": dim, "sinks": sinks, "tensors": tensors, "dout_fp32": dout_fp32, "fixed_dq": fixed_dq}


def _packed(name, docs, ratio, window, hq, hkv, sinks=0):
    return {"name": name, "kind": "packed", "docs": ",".join(str(t) for t in docs), "ratio": ratio, "window": window,
            "hq": hq, "hkv": hkv, "sinks": sinks}


def _prefill(name, kind, batch, raw_len, ratio, window, hq, hkv, sinks=0, chunk_units=0):
    return {"name": name, "kind": kind, "batch": batch, "raw_len": raw_len, "ratio": ratio, "window": window, "hq": hq,
            "hkv": hkv, "sinks": sinks, "chunk_units": chunk_units}


def _decode(name, seqs, max_len, min_len, hq, hkv, static=False):
    return {"name": name, "kind": "decode", "seqs": seqs, "max_len": max_len, "min_len": min_len, "hq": hq, "hkv": hkv,
            "static": static}


def _loop(name, batch, raw_len, ratio, window, hq, hkv, sinks=0):
    return {"name": name, "kind": "loop", "batch": batch, "raw_len": raw_len, "ratio": ratio, "window": window, "hq": hq,
            "hkv": hkv, "sinks": sinks}


def listed():
    return [
        # one interactive user's token over a short compressed cache: all latency
        _decode("decode_single_short", 1, 1337, 1337, 32, 8),
        # a serving batch whose requests have come to different lengths
        _decode("decode_ragged_batch", 17, 6000, 150, 32, 8),
        # the repository's decode workload: 64 sequences of 8192 gists and a 1024-token window, memory-bound
        _decode("decode_cache", 64, 9216, 9216, 32, 8),
        # generation itself, eight requests in step: append and attend for two gist units of 8 raw tokens and their gists
        _loop("decode_loop", 8, 8192, 8, 1024, 32, 8),
        # the repository's smallest training problem (one head, head_dim 64, fp32 dO): launches and latency
        _train("train_tiny", 1, 448, 7, 64, 1, 1, 64, tensors="shifted", dout_fp32=True),
        # one layer of an 8B-parameter model on one 16K sample
        _train("llama8b_layer", 1, 16384, 8, 1024, 32, 8, 128),
        # the repository's training batch: the largest case
        _train("train_batch", 4, 32768, 4, 2048, 32, 8, 128),
        # a multi-head layer with 128 sinks and the short window, rotary embedding included (the speed-table shape)
        _train("mha_sinks_rope", 1, 16384, 4, 128, 32, 32, 128, sinks=128, tensors="rope"),
        # a head_dim-64 model with a ratio that does not divide the tile, tensors shifted explicitly
        _train("head64_ratio7", 2, 8190, 7, 700, 16, 4, 64, sinks=5, tensors="shifted"),
        # a packed sample: documents of very different lengths, a few of them equal
        _packed("packed_docs", [8192, 3848, 3848, 1800, 1024, 1024, 1024, 408, 64], 8, 1024, 32, 8, sinks=4),
        # a 128K prompt in one pass, then its compaction
        _prefill("long_prefill", "prefill", 1, 131072, 16, 4096, 32, 8),
        # a 48K prompt (ragged last chunk) encoded in chunks of 8192 raw tokens over the compressed cache
        _prefill("chunked_prefill", "chunks", 1, 48 * 1024 + 16 * 37, 16, 4096, 32, 8, chunk_units=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds above at other sizes; never more work than the largest listed case."""
    kind = rng.choice(["decode", "decode", "loop", "train", "train", "train", "packed", "prefill", "chunks"])
    hq, hkv = rng.choice([(32, 8), (32, 8), (16, 4), (32, 32), (16, 2), (12, 4)])
    if kind == "decode":
        seqs = _log_int(rng, 1, 64)
        longest = _log_int(rng, 200, 9216)
        shortest = longest if rng.random() < 0.5 else rng.randint(1, longest)
        c = _decode(None, seqs, longest, shortest, hq, hkv)
        c["static"] = seqs <= 8 and rng.random() < 0.25
    elif kind == "loop":
        ratio = rng.choice([4, 8, 8, 16])
        c = _loop(None, _log_int(rng, 1, 32), ratio * _log_int(rng, 32, 2048), ratio, rng.choice([128, 512, 1024, 2048]), hq, hkv,
                  sinks=rng.choice([0, 0, 4, 128]))
    elif kind in ("prefill", "chunks"):
        ratio = rng.choice([4, 8, 16])
        units = _log_int(rng, 256, 65536 // ratio)
        c = _prefill(None, kind, 1, ratio * units, ratio, rng.choice([128, 1024, 4096]), hq, hkv, sinks=rng.choice([0, 0, 4, 128]),
                     chunk_units=max(1, -(-units // rng.randint(2, 8))) if kind == "chunks" else 0)
    elif kind == "packed":
        ratio = rng.choice([4, 8, 16])
        docs = [ratio * _log_int(rng, 4, 8192 // ratio) for _ in range(rng.randint(2, 12))]
        if rng.random() < 0.5:
            docs += [docs[-1]] * rng.randint(1, 3)
        c = _packed(None, docs, ratio, rng.choice([128, 512, 1024]), hq, hkv, sinks=rng.choice([0, 0, 4]))
    else:
        tensors = rng.choice(["interleaved", "interleaved", "rope", "shifted"])
        dim = rng.choice([64, 128]) if tensors == "shifted" else 128
        ratio = rng.choice([3, 5, 7, 8]) if tensors == "shifted" else rng.choice([2, 4, 8, 16])
        batch = rng.choice([1, 1, 2, 3])
        c = _train(None, batch, ratio * _log_int(rng, 256 // ratio, 24576 // (batch * ratio)), ratio,
                   rng.choice([64, 128, 1000, 1024, 2048]), hq, hkv, dim, sinks=rng.choice([0, 0, 5, 128]), tensors=tensors,
                   dout_fp32=rng.random() < 0.2, fixed_dq=tensors == "shifted" and rng.random() < 0.25)
    del c["name"]
    return c


# ----------------------------------------------------------------------------------------------------------------
# What is visible (for the operation counts): every token sees the sinks, the earlier gists and the raw tokens of
# its unit and the k units before it.
def _lens(case, raw_len=None):
    t = case["raw_len"] if raw_len is None else raw_len
    r, s = case["ratio"], case["sinks"]
    n = t // r
    k = min(-(-case["window"] // r), n)
    return s, t, r, n, k


def _pairs(case, raw_len=None):
    s, t, r, n, k = _lens(case, raw_len)
    in_window = k * (k - 1) // 2 + (n - k) * k  # sum over units of min(unit, k)
    before = n * (n - 1) // 2
    raw = r * r * in_window + n * (r * (r + 1) // 2) + r * before
    gist = r * (in_window + n) + before + n
    return s * (s + 1) // 2 + s * (t + n) + raw + gist


def _tokens(case, raw_len=None):
    s, t, _, n, _ = _lens(case, raw_len)
    return s + t + n


def _compact_len(case):
    s, _, r, n, k = _lens(case)
    return s + n + k * r


def _decode_lens(case):
    """The sequences' lengths: spread evenly from the longest to the shortest."""
    m = case["seqs"]
    return [case["max_len"] - (case["max_len"] - case["min_len"]) * i // max(1, m - 1) for i in range(m)]


def work(case):
    kind, hq, hkv = case["kind"], case["hq"], case["hkv"]
    if kind == "decode":
        cached = sum(_decode_lens(case))
        return {"bytes": cached * hkv * 512 + case["seqs"] * hq * (512 + 4), "flops": 4 * 128 * cached * hq}
    if kind == "loop":
        r, steps = case["ratio"], 2 * (case["ratio"] + 1)
        evicted = r if case["raw_len"] // r >= -(-case["window"] // r) else 0  # when the second unit opens
        entries = sum(_compact_len(case) + i + 1 - (evicted if i > r else 0) for i in range(steps)) * case["batch"]
        return {"bytes": entries * hkv * 512 + case["batch"] * steps * (hq * 516 + hkv * 1024), "flops": 4 * 128 * entries * hq}
    if kind in ("prefill", "chunks"):
        n = _tokens(case) * case["batch"]
        kept = _compact_len(case) * case["batch"] * hkv * 512
        return {"bytes": n * (hq * (512 + 4) + hkv * 512) + kept, "flops": 4 * 128 * _pairs(case) * hq * case["batch"]}
    if kind == "packed":
        docs = [int(t) for t in case["docs"].split(",")]
        n, pairs = sum(_tokens(case, t) for t in docs), sum(_pairs(case, t) for t in docs)
        return {"bytes": n * (hq * (4 * 256 + 4) + hkv * 4 * 256), "flops": 14 * 128 * pairs * hq}
    n, d = _tokens(case) * case["batch"], case["dim"]
    dout = 4 if case["dout_fp32"] else 2
    return {"bytes": n * (hq * (d * (6 + dout) + 4) + hkv * 8 * d), "flops": 14 * d * _pairs(case) * hq * case["batch"]}


def tolerance(case):
    # bf16 probabilities (and bf16 dS), fp32 sums, bf16 results.  Against the same attention in fp64 the worst output
    # measured, as relative 2-norm and as the largest difference over max(rms, value): decode 2.2e-3 and 0.009, a whole
    # sequence's forward 2.2e-3 and 0.027, gradients 2.5e-3 and 0.07.  Four times that.
    if case["kind"] in ("decode", "loop"):
        return {"rel": 9e-3, "max": 0.036}
    return {"rel": 9e-3, "max": 0.11} if case["kind"] in ("prefill", "chunks") else {"rel": 1e-2, "max": 0.28}


# ----------------------------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _randn(g, *shape, dtype=torch.bfloat16):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32).to(dtype)


def _bytes(n):
    return torch.empty(max(int(n), 16), dtype=torch.uint8, device=DEV)


def _pages(g, seqs, per_seq, hkv, fill):
    """A paged cache whose sequences' pages lie in random order, and its block table."""
    blocks = seqs * per_seq
    shape = (blocks, hkv, PAGE, 128)
    make = (lambda: torch.randn(shape, generator=g, device=DEV, dtype=torch.bfloat16)) if fill else \
           (lambda: torch.zeros(shape, device=DEV, dtype=torch.bfloat16))
    table = torch.randperm(blocks, generator=g, device=DEV).to(torch.int32).reshape(seqs, per_seq)
    return make(), make(), table


def prepare(case, seed):
    return {"decode": _prepare_decode, "loop": _prepare_loop, "train": _prepare_train, "packed": _prepare_packed,
            "prefill": _prepare_prefill, "chunks": _prepare_chunks}[case["kind"]](case, seed)


def run(st):
    return st["run"](st)


def _prepare_decode(case, seed):
    g, seqs, hq, hkv = _gen(seed), case["seqs"], case["hq"], case["hkv"]
    per_seq = -(-case["max_len"] // PAGE)
    kc, vc, table = _pages(g, seqs, per_seq, hkv, True)
    st = {"run": _run_decode_static if case["static"] else _run_decode, "kc": kc, "vc": vc, "table": table,
          "lens": torch.tensor(_decode_lens(case), dtype=torch.int32, device=DEV), "q": _randn(g, seqs, hq, 128),
          "o": torch.empty(seqs, hq, 128, dtype=torch.bfloat16, device=DEV),
          "lse": torch.empty(seqs, hq, dtype=torch.float32, device=DEV)}
    if not case["static"]:
        st["ws"] = _bytes(ug.unigist_decode_workspace_bytes(seqs, hq, hkv, 128, per_seq))
    return st


def _run_decode(st):
    ug.unigist_decode(st["q"], st["kc"], st["vc"], st["table"], st["lens"], st["o"], st["lse"], st["ws"])
    return st["o"], st["lse"]


def _run_decode_static(st):
    ug.unigist_decode_static(st["q"], st["kc"], st["vc"], st["table"], st["lens"], st["o"], st["lse"])
    return st["o"], st["lse"]


def _prepare_loop(case, seed):
    g, b, hq, hkv, r = _gen(seed), case["batch"], case["hq"], case["hkv"], case["ratio"]
    steps = 2 * (r + 1)
    p = ug.Problem(b, case["raw_len"], r, case["window"], hq, hkv, 128, num_sinks=case["sinks"])
    length = _compact_len(case)
    per_seq = -(-(length + steps) // PAGE)
    kc, vc, table = _pages(g, b, per_seq, hkv, True)
    return {"run": _run_loop, "p": p, "units": case["raw_len"] // r, "kc": kc, "vc": vc, "table": table,
            "prompt_lens": torch.full((b,), length, dtype=torch.int32, device=DEV),
            "lens": torch.empty(b, dtype=torch.int32, device=DEV),
            "state": torch.zeros(ug.unigist_cache_state_bytes(p) // 4, dtype=torch.int32, device=DEV),
            # every token has its own rows, as a model hands them over
            "q": list(_randn(g, steps, b, hq, 128)), "k": list(_randn(g, steps, b, hkv, 128)),
            "v": list(_randn(g, steps, b, hkv, 128)),
            "o": list(torch.empty(steps, b, hq, 128, dtype=torch.bfloat16, device=DEV)),
            "lse": list(torch.empty(steps, b, hq, dtype=torch.float32, device=DEV)),
            "ws": _bytes(ug.unigist_decode_workspace_bytes(b, hq, hkv, 128, per_seq))}


def _run_loop(st):
    p = st["p"]
    st["lens"].copy_(st["prompt_lens"])  # the cache as prefill left it
    ug.unigist_cache_state_init(p, st["units"], st["state"])
    for i, (q, k, v, o, lse) in enumerate(zip(st["q"], st["k"], st["v"], st["o"], st["lse"])):
        ug.unigist_cache_append(p, k, v, i % (p.ratio + 1) == p.ratio, st["kc"], st["vc"], st["table"], st["lens"], st["state"])
        ug.unigist_decode_step(p, q, st["kc"], st["vc"], st["table"], st["lens"], st["state"], o, lse, st["ws"])
    return st["o"], st["lse"], st["lens"], st["kc"], st["vc"]


def _prepare_train(case, seed):
    g, b, hq, hkv, d = _gen(seed), case["batch"], case["hq"], case["hkv"], case["dim"]
    flags = (ug.FLAG_DOUT_FP32 if case["dout_fp32"] else 0) | (ug.FLAG_INTERLEAVED if case["tensors"] == "interleaved" else 0)
    flags |= ug.FLAG_DETERMINISTIC_DQ if case["fixed_dq"] else 0
    p = ug.Problem(b, case["raw_len"], case["ratio"], case["window"], hq, hkv, d, num_sinks=case["sinks"], flags=flags)
    n = _tokens(case)
    st = {"run": {"interleaved": _run_train, "shifted": _run_train_shifted, "rope": _run_train_rope}[case["tensors"]], "p": p,
          "q": _randn(g, b, n, hq, d), "k": _randn(g, b, n, hkv, d), "v": _randn(g, b, n, hkv, d),
          "do": _randn(g, b, n, hq, d, dtype=torch.float32 if case["dout_fp32"] else torch.bfloat16),
          "lse": torch.empty(b, hq, n, dtype=torch.float32, device=DEV), "ws": _bytes(ug.unigist_workspace_bytes(p, ug.OP_BWD))}
    for name, like in (("o", "q"), ("dq", "q"), ("dk", "k"), ("dv", "v")):
        st[name] = torch.empty_like(st[like])
    if case["tensors"] != "interleaved":  # shifted copies of everything, as a program without the fused addressing keeps
        for name in ("q", "k", "v", "do", "o", "dq", "dk", "dv"):
            st[name + "_s"] = torch.empty_like(st[name])
    return st


def _run_train(st):
    p = st["p"]
    ug.unigist_attn_fwd(p, st["q"], st["k"], st["v"], st["o"], st["lse"])
    ug.unigist_attn_bwd(p, st["q"], st["k"], st["v"], st["o"], st["lse"], st["do"], st["dq"], st["dk"], st["dv"], st["ws"])
    return st["o"], st["lse"], st["dq"], st["dk"], st["dv"]


def _attend_shifted(st):
    p = st["p"]
    ug.unigist_attn_fwd(p, st["q_s"], st["k_s"], st["v_s"], st["o_s"], st["lse"])
    ug.unigist_gist_unshift(p, st["o_s"], st["o"])
    ug.unigist_gist_shift(p, st["do"], st["do_s"])
    ug.unigist_attn_bwd(p, st["q_s"], st["k_s"], st["v_s"], st["o_s"], st["lse"], st["do_s"], st["dq_s"], st["dk_s"], st["dv_s"],
                        st["ws"])


def _run_train_shifted(st):
    p = st["p"]
    for name in ("q", "k", "v"):
        ug.unigist_gist_shift(p, st[name], st[name + "_s"])
    _attend_shifted(st)
    for name in ("dq", "dk", "dv"):
        ug.unigist_gist_unshift(p, st[name + "_s"], st[name])
    return st["o"], st["lse"], st["dq"], st["dk"], st["dv"]


def _run_train_rope(st):
    p = st["p"]
    for name in ("q", "k"):
        ug.unigist_rope(p, st[name], st[name + "_s"], ROPE_BASE, ug.ROPE_TO_SHIFTED)
    ug.unigist_gist_shift(p, st["v"], st["v_s"])
    _attend_shifted(st)
    for name in ("dq", "dk"):
        ug.unigist_rope(p, st[name + "_s"], st[name], ROPE_BASE, ug.ROPE_FROM_SHIFTED | ug.ROPE_INVERSE)
    ug.unigist_gist_unshift(p, st["dv_s"], st["dv"])
    return st["o"], st["lse"], st["dq"], st["dk"], st["dv"]


def _prepare_packed(case, seed):
    g, hq, hkv = _gen(seed), case["hq"], case["hkv"]
    docs = [int(t) for t in case["docs"].split(",")]
    p = ug.Problem(1, docs[0], case["ratio"], case["window"], hq, hkv, 128, num_sinks=case["sinks"], flags=ug.FLAG_INTERLEAVED)
    n = ug.unigist_docs_total_len(p, docs)
    st = {"run": _run_packed, "p": p, "docs": docs, "q": _randn(g, n, hq, 128), "k": _randn(g, n, hkv, 128),
          "v": _randn(g, n, hkv, 128), "do": _randn(g, n, hq, 128), "lse": torch.empty(hq * n, dtype=torch.float32, device=DEV),
          "ws": _bytes(ug.unigist_docs_workspace_bytes(p, ug.OP_BWD, docs))}
    for name, like in (("o", "q"), ("dq", "q"), ("dk", "k"), ("dv", "v")):
        st[name] = torch.empty_like(st[like])
    return st


def _run_packed(st):
    p, docs = st["p"], st["docs"]
    ug.unigist_attn_fwd_docs(p, docs, st["q"], st["k"], st["v"], st["o"], st["lse"])
    ug.unigist_attn_bwd_docs(p, docs, st["q"], st["k"], st["v"], st["o"], st["lse"], st["do"], st["dq"], st["dk"], st["dv"], st["ws"])
    return st["o"], st["lse"], st["dq"], st["dk"], st["dv"]


def _prompt_cache(g, case):
    per_seq = -(-_compact_len(case) // PAGE)
    kc, vc, table = _pages(g, case["batch"], per_seq, case["hkv"], False)
    return {"kc": kc, "vc": vc, "table": table, "lens": torch.zeros(case["batch"], dtype=torch.int32, device=DEV)}


def _prepare_prefill(case, seed):
    g, b, hq, hkv = _gen(seed), case["batch"], case["hq"], case["hkv"]
    n = _tokens(case)
    p = ug.Problem(b, case["raw_len"], case["ratio"], case["window"], hq, hkv, 128, num_sinks=case["sinks"], flags=ug.FLAG_INTERLEAVED)
    return {"run": _run_prefill, "p": p, "q": _randn(g, b, n, hq, 128), "k": _randn(g, b, n, hkv, 128),
            "v": _randn(g, b, n, hkv, 128), "o": torch.empty(b, n, hq, 128, dtype=torch.bfloat16, device=DEV),
            "lse": torch.empty(b, hq, n, dtype=torch.float32, device=DEV), **_prompt_cache(g, case)}


def _run_prefill(st):
    p = st["p"]
    ug.unigist_attn_fwd(p, st["q"], st["k"], st["v"], st["o"], st["lse"])
    ug.unigist_kv_compact(p, st["k"], st["v"], st["kc"], st["vc"], st["table"], st["lens"])
    return st["o"], st["lse"], st["kc"], st["vc"], st["lens"]


def _prepare_chunks(case, seed):
    g, b, hq, hkv, r = _gen(seed), case["batch"], case["hq"], case["hkv"], case["ratio"]
    p = ug.Problem(b, case["raw_len"], r, case["window"], hq, hkv, 128, num_sinks=case["sinks"])
    units, chunks, need = case["raw_len"] // r, [], 16
    for u0 in range(0, units, case["chunk_units"]):
        c = min(case["chunk_units"], units - u0)
        n = (case["sinks"] if u0 == 0 else 0) + c * (r + 1)
        chunks.append((u0, c, _randn(g, b, n, hq, 128), _randn(g, b, n, hkv, 128), _randn(g, b, n, hkv, 128),
                       torch.empty(b, n, hq, 128, dtype=torch.bfloat16, device=DEV),
                       torch.empty(b, hq, n, dtype=torch.float32, device=DEV)))
        need = max(need, ug.unigist_prefill_workspace_bytes(p, u0, c))
    return {"run": _run_chunks, "p": p, "chunks": chunks, "ws": _bytes(need), **_prompt_cache(g, case)}


def _run_chunks(st):
    for u0, c, q, k, v, o, lse in st["chunks"]:
        ug.unigist_prefill_chunk(st["p"], u0, c, q, k, v, st["kc"], st["vc"], st["table"], st["lens"], o, lse, st["ws"])
    return [x[5] for x in st["chunks"]], [x[6] for x in st["chunks"]], st["kc"], st["vc"], st["lens"]


# ----------------------------------------------------------------------------------------------------------------
# The same results in 64 bits, from the definition: torch alone, on the sequence as it is (no gist shift, no tiles).
def exact(case, seed):
    st = prepare(case, seed)  # for the inputs
    return {"decode": _exact_decode, "loop": _exact_loop, "train": _exact_train, "packed": _exact_packed,
            "prefill": _exact_prefill, "chunks": _exact_chunks}[case["kind"]](case, st)


def _one_query64(q, k, v):
    """q [Hq, 128] over k, v [Hkv, tokens, 128]."""
    hkv = k.shape[0]
    s = torch.einsum("hgd,htd->hgt", q.double().reshape(hkv, -1, 128), k.double()) / math.sqrt(128)
    lse = torch.logsumexp(s, -1)
    return torch.einsum("hgt,htd->hgd", (s - lse[..., None]).exp(), v.double()).reshape(-1, 128), lse.reshape(-1)


def _cached(pages, row, length):
    """The first `length` tokens of one sequence: [Hkv, length, 128]."""
    return pages[row.long()].transpose(0, 1).flatten(1, 2)[:, :length]


def _exact_decode(case, st):
    rows = [_one_query64(st["q"][i], _cached(st["kc"], st["table"][i], n), _cached(st["vc"], st["table"][i], n))
            for i, n in enumerate(_decode_lens(case))]
    return torch.stack([o for o, _ in rows]), torch.stack([lse for _, lse in rows])


def _exact_loop(case, st):
    s, _, r, n, _ = _lens(case)
    length, steps = _compact_len(case), len(st["q"])
    live = torch.ones(steps, length + steps, dtype=torch.bool, device=DEV).tril(length)
    if n >= -(-case["window"] // r):  # the second unit's first token: the oldest unit of the window is gone
        live[r + 1:, s + n:s + n + r] = False
    o, lse = [], []
    for b in range(case["batch"]):
        k, v = (torch.cat([_cached(st[pages], st["table"][b], length)] + [x[b][:, None] for x in st[new]], 1)
                for pages, new in (("kc", "k"), ("vc", "v")))
        rows = [_one_query64(st["q"][i][b], k[:, live[i]], v[:, live[i]]) for i in range(steps)]
        o.append([x for x, _ in rows])
        lse.append([x for _, x in rows])
    return [torch.stack(x) for x in zip(*o)], [torch.stack(x) for x in zip(*lse)], None, None, None


def _kinds(case, raw_len, device=DEV):
    """Of every token of a sequence: its unit (-1: a sink) and whether it is a gist; and the shifted order's tokens."""
    s, t, r, n, _ = _lens(case, raw_len)
    i = torch.arange(s + t + n, device=device) - s
    unit = torch.where(i < 0, -1, i // (r + 1))
    gist = (i >= 0) & (i % (r + 1) == r)
    return unit, gist, torch.argsort(gist, stable=True)


def _sequence64(case, q, k, v, do=None, raw_len=None):
    """One sequence, q, do [N, Hq, D], k, v [N, Hkv, D] -> o [N, Hq, D], lse [Hq, N] in shifted order, and with do the
    gradients dq, dk, dv."""
    s, _, r, _, w = _lens(case, raw_len)
    unit, gist, order = _kinds(case, raw_len)
    (total, hq, d), hkv, scale = q.shape, k.shape[1], 1 / math.sqrt(q.shape[2])
    out = {name: torch.zeros(x.shape, dtype=torch.float64, device=DEV)
           for name, x in (("o", q), ("dq", q), ("dk", k), ("dv", v)) if do is not None or name == "o"}
    lse = torch.empty(hq, total, dtype=torch.float64, device=DEV)
    at = torch.arange(total, device=DEV)
    for a in range(0, total, 1024):
        rows = at[a:a + 1024]
        first = max((a - s) // (r + 1) - w, 0)  # the first unit whose raw tokens the block's first row sees
        cols = at[:rows[-1] + 1]
        cols = cols[(unit[cols] < 0) | gist[cols] | (unit[cols] >= first)]
        seen = (cols <= rows[:, None]) & ((unit[cols] < 0) | gist[cols] | (unit[cols] >= unit[rows][:, None] - w))
        for h in range(hkv):
            heads = slice(h * hq // hkv, (h + 1) * hq // hkv)
            qh = q[rows, heads].double().transpose(0, 1)
            kh, vh = k[cols, h].double(), v[cols, h].double()
            p = (qh @ kh.T * scale).masked_fill_(~seen, -math.inf)
            norm = torch.logsumexp(p, -1)
            lse[heads, rows] = norm
            p = p.sub_(norm[..., None]).exp_()
            oh = p @ vh
            out["o"][rows, heads] = oh.transpose(0, 1)
            if do is not None:
                doh = do[rows, heads].double().transpose(0, 1)
                out["dv"][cols, h] += p.flatten(0, 1).T @ doh.flatten(0, 1)
                p *= (doh @ vh.T).sub_((doh * oh).sum(-1, keepdim=True))
                out["dq"][rows, heads] = (p @ kh * scale).transpose(0, 1)
                out["dk"][cols, h] += p.flatten(0, 1).T @ qh.flatten(0, 1) * scale
    return (out["o"], lse[:, order]) + ((out["dq"], out["dk"], out["dv"]) if do is not None else ())


def _rotated64(case, x, sign):
    """x [N, H, D]: feature j of the first half pairs with j + D / 2; a gist has the position of the raw token after it."""
    s, _, r, _, _ = _lens(case)
    unit, gist, _ = _kinds(case, case["raw_len"])
    i = torch.arange(len(unit), device=DEV)
    pos = torch.where(gist, s + (unit + 1) * r, i - unit.clamp_min(0)).double()
    half = x.shape[2] // 2
    angle = sign * pos[:, None, None] * ROPE_BASE ** (-torch.arange(half, device=DEV, dtype=torch.float64) / half)
    a, b = x.double().split(half, 2)
    return torch.cat([a * angle.cos() - b * angle.sin(), b * angle.cos() + a * angle.sin()], 2)


def _exact_train(case, st):
    rope, outs = case["tensors"] == "rope", []
    for b in range(case["batch"]):
        q, k = ((_rotated64(case, st[x][b], 1) if rope else st[x][b]) for x in ("q", "k"))
        o, lse, dq, dk, dv = _sequence64(case, q, k, st["v"][b], st["do"][b])
        if rope:
            dq, dk = _rotated64(case, dq, -1), _rotated64(case, dk, -1)
        outs.append((o, lse, dq, dk, dv))
    return tuple(torch.stack(x) for x in zip(*outs))


def _exact_packed(case, st):
    outs, a = [], 0
    for t in st["docs"]:
        b = a + _tokens(case, t)
        o, lse, dq, dk, dv = _sequence64(case, *(st[x][a:b] for x in ("q", "k", "v", "do")), raw_len=t)
        outs.append((o, lse.flatten(), dq, dk, dv))
        a = b
    return tuple(torch.cat(x) for x in zip(*outs))


def _exact_prefill(case, st):
    outs = [_sequence64(case, st["q"][b], st["k"][b], st["v"][b]) for b in range(case["batch"])]
    return torch.stack([o for o, _ in outs]), torch.stack([lse for _, lse in outs]), None, None, None


def _exact_chunks(case, st):
    s, t, r, _, _ = _lens(case)
    order = _kinds(case, t)[2]  # the tokens in the order [sinks | raw | gists]
    tokens, outs = [], []  # each chunk's tokens, in its own order of the same form
    for u0, c, *_ in st["chunks"]:
        tokens.append(torch.cat([order[:s if u0 == 0 else 0], order[s + u0 * r:s + (u0 + c) * r], order[s + t + u0:s + t + u0 + c]]))
    place = torch.argsort(torch.cat(tokens))
    for b in range(case["batch"]):
        q, k, v = (torch.cat([x[j][b] for x in st["chunks"]])[place] for j in (2, 3, 4))
        o, lse = _sequence64(case, q, k, v)
        by_token = torch.empty_like(lse)
        by_token[:, order] = lse
        outs.append(([o[i] for i in tokens], [by_token[:, i] for i in tokens]))
    return ([torch.stack(x) for x in zip(*(o for o, _ in outs))], [torch.stack(x) for x in zip(*(l for _, l in outs))], None,
            None, None)
