"""The work this library is measured on: one pass of one attention layer over one chunk of queries.

Every case goes through the public entry points of `paper_2602_08722_b200.api` the way a serving program calls them.
A case is a dict of plain values:

    entry      "prefill"  quoka_prefill_chunk, the chunk's keys and values already in the cache
               "append"   quoka_append_kv, then quoka_prefill_chunk (the loop of Algorithm 2)
               "dense"    quoka_dense_chunk_attn (a layer or chunk that is kept dense)
               "host"     quoka_prefill_chunk_host (the chunk lives in pinned host memory)
    batch, n_q, n_kv, d, dtype            the layer
    chunk                                 queries per sequence (1 = a generation step)
    ctx_len, ctx_min                      longest / shortest cached length of the batch
    max_ctx                               upper bound on the cached length the buffers are laid out for
    n_retain, kv_budget, budget_frac      retained queries; key budget in keys, or (0) as a fraction of the cached length
    paged                                 64-row pages in random order with a block table
    norms                                 inverse key norms kept beside the cache
"""
from __future__ import annotations

import math

import torch

from paper_2602_08722_b200 import api

PAGE = 64
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, **kw):
    c = {"name": name, "entry": "prefill", "batch": 1, "n_q": 32, "n_kv": 8, "d": 128, "dtype": "bf16", "chunk": 2048,
         "ctx_len": 32768, "ctx_min": 0, "max_ctx": 0, "n_retain": 128, "kv_budget": 0, "budget_frac": 0.12,
         "paged": False, "norms": False}
    c.update(kw)
    c["ctx_min"] = c["ctx_min"] or c["ctx_len"]
    c["max_ctx"] = c["max_ctx"] or c["ctx_len"]
    return c


def listed():
    return [
        # generation steps: one query per sequence.  A short conversation (latency of the launches), a long one, and a
        # batch of a paged serving mix with the norms of the cached keys kept.
        _case("decode_4k", entry="append", chunk=1, ctx_len=4003, max_ctx=4096, n_retain=16, kv_budget=256),
        _case("decode_32k", entry="append", chunk=1, ctx_len=32768, n_retain=16, kv_budget=256),
        _case("decode_mix_b16", entry="append", batch=16, chunk=1, ctx_len=32768, ctx_min=8192, n_retain=16, kv_budget=256,
              paged=True, norms=True),
        # the smallest layer of the tests, in both data types
        _case("tiny_bf16", n_q=8, n_kv=2, chunk=256, ctx_len=4096, n_retain=32, kv_budget=512),
        _case("tiny_f32", n_q=8, n_kv=2, chunk=256, ctx_len=4096, n_retain=32, kv_budget=512, dtype="f32"),
        # the paper's own chunk length, in the middle of a 32K prompt whose cache is laid out in full
        _case("chunk128_mid_32k", entry="append", chunk=128, ctx_len=19968, max_ctx=32768, n_retain=128),
        # odd sizes everywhere, head_dim 64, eight query heads per KV head, a quarter of the keys
        _case("ragged_d64", n_kv=4, d=64, chunk=777, ctx_len=20011, n_retain=50, budget_frac=0.25),
        # the benchmark's default: one 2048-token chunk at 32K
        _case("chunk2048_32k", n_retain=128, kv_budget=3932),
        # the same chunk from and to pinned host memory
        _case("chunk2048_32k_host", entry="host", n_retain=128, kv_budget=3932),
        # prefill of a paged serving batch, 8K to 64K cached
        _case("serving_mix", batch=8, chunk=1024, ctx_len=65536, ctx_min=8192, n_retain=64, paged=True),
        # the longest context
        _case("chunk4096_128k", chunk=4096, ctx_len=131072, n_retain=256, kv_budget=15729),
        # a chunk attended densely, as the layers or chunks outside the sparse path are
        _case("dense_2048_32k", entry="dense"),
    ]


# ----------------------------------------------------------------------------------------------- drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Rough cost of a case, in tensor-core flops: what keeps a drawn case below the largest listed one."""
    rows = -(-c["chunk"] // 256) * 256 if c["chunk"] > 1 else 1
    keys = sum((t if c["entry"] == "dense" else _budget(c, t)) + c["chunk"] / 2 for t in _ctx_lens(c))
    attn = 4.0 * c["n_q"] * rows * c["d"] * keys
    score = 2.0 * c["n_kv"] * min(c["n_retain"], c["chunk"]) * c["d"] * sum(_ctx_lens(c))
    return (attn + score) * (1.0 if c["d"] == 128 else 2.0) * (1.0 if c["dtype"] == "bf16" else 500.0)


def _state_bytes(c):
    return 2 * sum(t + c["chunk"] for t in _ctx_lens(c)) * c["n_kv"] * c["d"] * (2 if c["dtype"] == "bf16" else 4)


def draw(rng):
    while True:
        kind = rng.choices(["prefill", "append", "decode", "dense", "host"], [9, 4, 6, 2, 1])[0]
        d = rng.choice([64, 128, 128])
        n_kv, group = rng.choice([(8, 4), (8, 4), (2, 4), (4, 8), (8, 1), (16, 2), (5, 3)])
        c = _case("", n_q=n_kv * group, n_kv=n_kv, d=d, paged=kind != "host" and rng.random() < 0.4,
                  norms=kind != "dense" and rng.random() < 0.2, ctx_len=_log_int(rng, 256, 131072))
        del c["name"]
        c["dtype"] = "f32" if rng.random() < 0.12 else "bf16"
        c["batch"] = rng.choice([1, 1, 1, 2, 3, 4, 8])
        if kind == "decode":
            c.update(entry="append", chunk=1, batch=rng.choice([1, 1, 2, 4, 8, 16]), n_retain=16,
                     kv_budget=_log_int(rng, 64, 4096))
        else:
            c.update(entry=kind, chunk=_log_int(rng, 128, 1024) if kind == "append" else _log_int(rng, 32, 4096))
            c["n_retain"] = rng.choice([16, 32, 64, 128, 256, 512, rng.randint(16, 512)])
            if rng.random() < 0.4:
                c["kv_budget"] = _log_int(rng, 256, 16384)
            else:
                c["budget_frac"] = rng.choice([0.05, 0.12, 0.12, 0.25, 0.5])
        c["ctx_min"] = max(1, int(c["ctx_len"] * rng.uniform(0.15, 1.0))) if c["batch"] > 1 else c["ctx_len"]
        c["max_ctx"] = c["ctx_len"] if rng.random() < 0.6 else int(c["ctx_len"] * rng.uniform(1.0, 1.5))
        if c["norms"] and kind == "host":
            c["norms"] = False                # the host-buffer call does not keep the norms of the rows it brings in
        if _cost(c) <= 1.1e12 and _state_bytes(c) <= 1.1e9:
            return c


# ----------------------------------------------------------------------------------------------- sizes of a case
def _ctx_lens(c):
    """Cached lengths of the batch: the longest first, the others spread over [ctx_min, ctx_len]."""
    lo, hi = c["ctx_min"], c["ctx_len"]
    return [hi - int((hi - lo) * ((s * 0.6180339887) % 1.0)) for s in range(c["batch"])]


def _budget(c, t):
    return min(c["kv_budget"], t) if c["kv_budget"] > 0 else min(t, int(c["budget_frac"] * t + 0.5))


# ----------------------------------------------------------------------------------------------- inputs
class _State:
    pass


def _keys(shape, dtype, g):
    """Keys ~ N(0, I), one position in twenty three times as long (independently per KV head)."""
    k = torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)
    big = torch.rand(shape[:-1], device="cuda", generator=g) < 0.05
    return k.mul_((1.0 + 2.0 * big.to(dtype)).unsqueeze(-1))


def prepare(case, seed):
    """Queries scattered around a mean direction per head, keys and values normal: the distributions of the tests."""
    c = case
    st = _State()
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = DTYPES[c["dtype"]]
    b, n_q, n_kv, d, C = c["batch"], c["n_q"], c["n_kv"], c["d"], c["chunk"]
    lens = _ctx_lens(c)
    mu = torch.randn(b, n_q, 1, d, device="cuda", generator=g)
    st.q = (mu + 0.7 * torch.randn(b, n_q, C, d, device="cuda", generator=g)).to(dt)
    st.ctx_len = torch.tensor(lens, dtype=torch.int32, device="cuda")
    table = None
    if c["paged"]:
        need = [-(-(t + C) // PAGE) for t in lens]
        perm = torch.randperm(sum(need), generator=torch.Generator().manual_seed(seed)).to(torch.int32)
        table = torch.full((b, -(-(c["max_ctx"] + C) // PAGE)), -1, dtype=torch.int32)
        off = 0
        for s, n in enumerate(need):
            table[s, :n] = perm[off:off + n]
            off += n
        table = table.cuda()
        shape = (sum(need), n_kv, PAGE, d)
    else:
        shape = (b, n_kv, c["max_ctx"] + C, d)
    st.table = table
    st.k = _keys(shape, dt, g)
    st.v = torch.empty(shape, dtype=dt, device="cuda").normal_(generator=g)
    st.out = torch.empty_like(st.q)
    st.p = api.make_params(st.q, st.k, st.out, st.ctx_len, n_retain=c["n_retain"], kv_budget=c["kv_budget"],
                           budget_frac=c["budget_frac"], max_ctx_len=c["max_ctx"], block_table=table)
    st.ws = api.alloc_workspace(st.p)
    st.norms = None
    if c["norms"]:
        st.norms = torch.zeros(shape[:3], dtype=torch.float32, device="cuda")
        api.quoka_update_key_norms(st.p, st.k, st.norms, True, st.ws)
        st.p.k_inv_norm = st.norms.data_ptr()
    if c["entry"] in ("append", "host"):
        st.k_new = _keys((b, n_kv, C, d), dt, g)
        st.v_new = torch.empty((b, n_kv, C, d), dtype=dt, device="cuda").normal_(generator=g)
    if c["entry"] == "host":
        st.ctx_host = torch.tensor(lens, dtype=torch.int32)
        st.q_host, st.k_new, st.v_new = (x.cpu().pin_memory() for x in (st.q, st.k_new, st.v_new))
        st.out_host = torch.empty(st.out.shape, dtype=dt, pin_memory=True)
    st.entry = c["entry"]
    return st


def run(st):
    if st.entry == "dense":
        api.quoka_dense_chunk_attn(st.p, st.q, st.k, st.v, st.out, None, st.ws)
        return {"out": st.out}
    if st.entry == "host":
        api.quoka_prefill_chunk_host(st.p, st.ctx_host, st.q_host, st.k_new, st.v_new, st.out_host, st.q, st.k, st.v,
                                     st.out, st.ws)
        torch.cuda.current_stream().synchronize()          # the caller reads the result on the host
        return {"out": st.out_host, "k": st.k, "v": st.v}
    if st.entry == "append":
        api.quoka_append_kv(st.p, st.k_new, st.v_new, st.k, st.v, st.norms, st.ws)
    api.quoka_prefill_chunk(st.p, st.q, st.k, st.v, st.out, None, None, st.ws)
    if st.entry == "append":
        res = {"out": st.out, "k": st.k, "v": st.v}
        if st.norms is not None:
            res["norms"] = st.norms
        return res
    return {"out": st.out}


# ----------------------------------------------------------------------------------------------- what a pass needs
def work(case):
    c = case
    es = 2 if c["dtype"] == "bf16" else 4
    n_q, n_kv, d, C = c["n_q"], c["n_kv"], c["d"], c["chunk"]
    N = min(c["n_retain"], C)
    nbytes = flops = 0.0
    for t in _ctx_lens(c):
        dense = c["entry"] == "dense"
        keys = t if dense else _budget(c, t)
        nbytes += 2 * n_q * C * d * es                                   # queries in, outputs out
        nbytes += n_kv * (t + C) * d * es + n_kv * (keys + C) * d * es   # every key once, the attended values once
        flops += 4.0 * n_q * C * d * (keys + (C + 1) / 2)
        if not dense:
            flops += 2.0 * n_kv * N * t * d + (4.0 * n_q * C * d if C > c["n_retain"] else 0.0)
        if c["entry"] in ("append", "host"):
            nbytes += 2 * n_kv * C * d * es                              # the new rows (written as they are read above)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Relative error of the output between two correct implementations of the same precision.

    Rounding alone (measured against the path in 64 bits on the same index lists): 2.3e-3 for bf16, 2.2e-7 for f32.
    The selection adds to it: two cosines, or two scores at the threshold, that lie within an ulp of each other may
    change places.  A key that changes places at the threshold alone cost at most 6.6e-3 (30 drawn cases, 6 seeds
    each); two retained queries that change ranks re-pair the heads of a group and replace some dozens of keys: nothing
    in most inputs, up to 7.3e-2 in 40 seeds of "ragged_d64" and 1.1e-1 in 12 of "chunk2048_32k", where a few long keys
    dominate some rows."""
    if case["entry"] == "dense":
        return {"rel": 1e-2 if case["dtype"] == "bf16" else 1e-5}
    return {"rel": 0.25 if case["chunk"] > case["n_retain"] else 2e-2}
