"""Parity of the CUDA path (through the C ABI) with the CPU oracle on the same seeded inputs."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import quoka_oracle as O
from paper_2602_08722_b200 import api, synth
from tests.parity import GpuProblem, attention_bound, check_attention, check_chain, check_query_ranks, f64, stratified_rows

pytestmark = pytest.mark.gpu

IMPLS = [pytest.param(api.IMPL_SIMT, id="simt"), pytest.param(api.IMPL_AUTO, id="auto")]


def problem(seed, *, batch=1, n_q=4, n_kv=2, d=128, T=1000, C=300, dtype="bf16", n_retain=24, kv_budget=177,
            budget_frac=0.0, impl=api.IMPL_AUTO, paged=False, capacity=None, max_ctx_len=None, score_mode="cosine",
            query_agg="max", cached_norms=False):
    inp = synth.make_chunk_inputs(seed, batch, n_q, n_kv, d, T, C, dtype, capacity=capacity)
    if paged:
        inp = synth.to_paged(inp, seed)
    return GpuProblem(inp, n_retain, kv_budget, budget_frac, impl=impl, paged=paged, max_ctx_len=max_ctx_len,
                      score_mode=score_mode, query_agg=query_agg, cached_norms=cached_norms)


# ---------------------------------------------------------------- small cases, every stage, all rows
@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("name", ["tiny_bf16", "tiny_f32"])
def test_tiny_config(name, impl):
    w = synth.WORKLOADS[name]
    gp = problem(1, n_q=w["n_q"], n_kv=w["n_kv"], d=w["d"], T=w["T"], C=w["C"], dtype=w["dtype"],
                 n_retain=w["n_retain"], kv_budget=w["kv_budget"], impl=impl)
    gp.run_staged()
    check_chain(gp)


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("d,dtype", [(128, "bf16"), (64, "bf16"), (128, "f32"), (64, "f32")])
def test_ragged_sizes(d, dtype, impl):
    # T, C, N, B all off tile boundaries; several 128-row tiles and a ragged tail everywhere
    gp = problem(2, n_q=6, n_kv=2, d=d, T=1237, C=333, dtype=dtype, n_retain=37, kv_budget=291, impl=impl)
    gp.run_staged()
    check_chain(gp)


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("T,C,n_retain,kv_budget", [
    (0, 200, 16, 64),        # empty cache: pure causal self-attention of the chunk
    (1, 130, 16, 64),        # one cached key
    (77, 129, 8, 500),       # budget covers the cache: identity selection, equals dense
    (500, 40, 64, 100),      # chunk not longer than N_Q: no query sub-selection
    (300, 1, 4, 50),         # single-query chunk
    (129, 257, 256, 128),    # N_Q just below C
])
def test_degenerate_cases(T, C, n_retain, kv_budget, impl):
    gp = problem(3, n_q=4, n_kv=2, T=T, C=C, n_retain=n_retain, kv_budget=kv_budget, impl=impl)
    gp.run_staged()
    check_chain(gp)
    if kv_budget >= T:
        q, k, v, _ = gp.oracle_inputs(0)
        dense, _ = O.dense_chunk_attention(q, k, v, T)
        check_attention(f64(gp.out[0]), dense, "bf16")


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("G", [1, 4, 8])
def test_gqa_ratios(G, impl):
    gp = problem(4, n_q=8, n_kv=8 // G, T=700, C=260, n_retain=32, kv_budget=0, budget_frac=0.25, impl=impl)
    gp.run_staged()
    check_chain(gp)


@pytest.mark.parametrize("n_q,n_kv", [(12, 2), (10, 5), (14, 7), (9, 3), (5, 5)])
def test_gqa_ratios_that_are_not_powers_of_two(n_q, n_kv):
    # clusters of pairs in three or four parts, tiles of 126 (six and three heads) and 128 rows
    gp = problem(960, batch=2, n_q=n_q, n_kv=n_kv, T=[4100, 200], C=129, n_retain=16, kv_budget=0, budget_frac=0.9)
    gp.run_staged()
    check_chain(gp)


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("paged", [False, True])
def test_batched_variable_lengths(paged, impl):
    gp = problem(5, batch=3, n_q=4, n_kv=2, T=[900, 130, 517], C=192, n_retain=16, kv_budget=0, budget_frac=0.12,
                 impl=impl, paged=paged)
    gp.run_staged()
    check_chain(gp)


def test_max_ctx_len_may_exceed_every_sequence():
    gp = problem(6, T=600, C=128, capacity=2048, max_ctx_len=1500, kv_budget=0, budget_frac=0.5)
    gp.run_staged()
    check_chain(gp)


# ---------------------------------------------------------------- generation phase: one query, no query sub-selection
@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("paged", [False, True])
def test_decode_step_single_query_per_sequence(paged, impl):
    # a chunk of one query: Alg. 1 skips the sub-selection (C <= N_Q), Qbar is the group mean of the
    # normalised query, the budget selects among the cached keys, the query attends them and itself
    gp = problem(15, batch=3, n_q=8, n_kv=2, T=[2100, 333, 1290], C=1, n_retain=16, kv_budget=128, impl=impl,
                 paged=paged)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(staged, gp.out)


def test_decode_step_full_size_32k():
    w = synth.WORKLOADS["decode_32k"]
    gp = problem(0, n_q=w["n_q"], n_kv=w["n_kv"], d=w["d"], T=w["T"], C=w["C"], n_retain=w["n_retain"],
                 kv_budget=w["kv_budget"])
    gp.run_staged()
    check_chain(gp)


@pytest.mark.parametrize("d,dtype", [(64, "bf16"), (128, "f32"), (64, "f32")])
def test_decode_step_other_layouts_and_dense(d, dtype):
    gp = problem(19, batch=2, n_q=8, n_kv=4, d=d, T=[1500, 77], C=1, dtype=dtype, n_retain=4, kv_budget=100)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(staged, gp.out)
    # the same query over every cached row (Eq. 2)
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    for s_ in range(gp.b):
        q, k, v, T = gp.oracle_inputs(s_)
        want, lse = O.dense_chunk_attention(q, k, v, T)
        check_attention(f64(gp.out[s_]), want, dtype)
        assert np.abs(f64(gp.lse[s_]) - lse).max() <= 2e-3


def test_decode_step_with_more_listed_rows_than_the_gather_kernel_holds():
    # 8500 listed rows + the query's own exceed the decode attention kernel's shared-memory logits: the general
    # attention kernel takes over, the matrix-vector scoring stays
    gp = problem(20, n_q=4, n_kv=2, T=9000, C=1, n_retain=4, kv_budget=8500)
    gp.run_staged()
    check_chain(gp)


# ---------------------------------------------------------------- cached inverse key norms
@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("paged", [False, True])
def test_cached_key_norms(paged, impl):
    gp = problem(16, batch=2, n_q=8, n_kv=2, T=[1700, 640], C=200, n_retain=24, kv_budget=0, budget_frac=0.2, impl=impl,
                 paged=paged, cached_norms=True)
    # the cache itself against the oracle, on every row that exists
    for s in range(gp.b):
        T = int(gp.inp.ctx_len[s])
        want = O.key_inv_norms(f64(gp.inp.k[s, :, : T + gp.C]))
        if paged:
            tbl = gp.inp.block_table[s]
            got = np.stack([f64(gp.k_inv_norm[int(tbl[t // 64]), :, t % 64]) for t in range(T + gp.C)], axis=1)
        else:
            got = f64(gp.k_inv_norm[s, :, : T + gp.C])
        np.testing.assert_allclose(got, want, rtol=2e-6)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(staged, gp.out)
    # appending: only the chunk's rows are rewritten
    before = gp.k_inv_norm.clone()
    gp.k_inv_norm.fill_(7.0)
    api.quoka_update_key_norms(gp.p, gp.k, gp.k_inv_norm, False, gp.ws)
    torch.cuda.synchronize()
    changed = gp.k_inv_norm != 7.0
    assert int(changed.sum()) == gp.b * gp.n_kv * gp.C
    assert torch.equal(gp.k_inv_norm[changed], before[changed])


# ---------------------------------------------------------------- ablation variants of the scoring step
@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("score_mode,query_agg", [("dot", "max"), ("cosine", "mean"), ("dot", "mean")])
def test_scoring_ablation_variants(score_mode, query_agg, dtype, impl):
    gp = problem(13, n_q=8, n_kv=2, T=1500, C=290, dtype=dtype, n_retain=40, kv_budget=300, impl=impl,
                 score_mode=score_mode, query_agg=query_agg)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(staged, gp.out)


def test_scoring_ablation_with_more_than_256_retained_queries():
    gp = problem(14, n_q=4, n_kv=2, T=900, C=700, n_retain=300, kv_budget=200, score_mode="dot", query_agg="mean")
    gp.run_staged()
    check_chain(gp)


# ---------------------------------------------------------------- dense kernel, fused call, determinism
@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_dense_chunk_attention(dtype, impl):
    gp = problem(7, n_q=4, n_kv=2, T=777, C=300, dtype=dtype, impl=impl)
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v, T = gp.oracle_inputs(0)
    want, lse = O.dense_chunk_attention(q, k, v, T)
    check_attention(f64(gp.out[0]), want, dtype)
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3


@pytest.mark.parametrize("impl", IMPLS)
@pytest.mark.parametrize("paged", [False, True])
def test_fused_call_equals_staged_calls(paged, impl):
    gp = problem(8, batch=2, n_q=8, n_kv=2, T=[1500, 700], C=256, n_retain=32, kv_budget=200, impl=impl, paged=paged)
    gp.run_staged()
    staged_out, staged_idx = gp.out.clone(), gp.k_idx.clone()
    gp.out.zero_()
    k_idx2 = torch.full_like(gp.k_idx, -9)
    k_cnt2 = torch.full_like(gp.k_cnt, -9)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, k_idx2, k_cnt2, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(k_idx2, staged_idx) and torch.equal(k_cnt2, gp.k_cnt)
    assert torch.equal(gp.out, staged_out)
    # and without the optional outputs
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged_out)
    assert api.quoka_last_device_status(gp.ws) == 0


def test_fused_call_with_empty_cache():
    gp = problem(9, T=0, C=150, n_retain=8, kv_budget=32)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    q, k, v, T = gp.oracle_inputs(0)
    want, _ = O.dense_chunk_attention(q, k, v, 0)
    check_attention(f64(gp.out[0]), want, "bf16")
    assert int(gp.k_cnt[0]) == 0


@pytest.mark.parametrize("impl", IMPLS)
def test_runs_are_bit_identical(impl):
    gp = problem(10, n_q=8, n_kv=2, T=3000, C=256, n_retain=32, kv_budget=300, impl=impl)
    gp.run_staged()
    first = [t.clone() for t in (gp.q_idx, gp.qbar, gp.scores, gp.k_idx, gp.out)]
    for _ in range(2):
        gp.run_staged()
        for a, b in zip(first, (gp.q_idx, gp.qbar, gp.scores, gp.k_idx, gp.out)):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("shape", [dict(n_q=8, n_kv=2, T=2000, C=256, n_retain=32, kv_budget=256),
                                   # large enough to be cut into four slices of KV groups that overlap their copies
                                   dict(n_q=32, n_kv=8, T=3000, C=2048, n_retain=64, kv_budget=700),
                                   dict(batch=2, n_q=12, n_kv=6, T=[1500, 800], C=1536, n_retain=64, kv_budget=300)],
                         ids=["small", "four-slices", "two-slices-batch-2"])
def test_host_buffer_entry_point_matches_device_entry_point(shape):
    gp = problem(11, **shape)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    want = gp.out.clone()
    C = shape["C"]
    Ts = [int(t) for t in gp.inp.ctx_len]
    q_host = gp.inp.q.contiguous().pin_memory()
    k_new = torch.stack([gp.inp.k[s, :, T:T + C] for s, T in enumerate(Ts)]).contiguous().pin_memory()
    v_new = torch.stack([gp.inp.v[s, :, T:T + C] for s, T in enumerate(Ts)]).contiguous().pin_memory()
    out_host = torch.zeros_like(q_host).pin_memory()
    for s, T in enumerate(Ts):
        gp.k[s, :, T:T + C].zero_()
        gp.v[s, :, T:T + C].zero_()
    q_dev = torch.zeros_like(gp.q)
    gp.out.zero_()
    ctx_host = gp.inp.ctx_len.clone()
    api.quoka_prefill_chunk_host(gp.p, ctx_host, q_host, k_new, v_new, out_host, q_dev, gp.k, gp.v, gp.out, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(out_host, want.cpu())


@pytest.mark.parametrize("dtype,n_q,n_kv,C", [
    ("f32", 32, 8, 2048), ("bf16", 32, 16, 1300), ("bf16", 30, 5, 1536), ("bf16", 16, 2, 2560), ("bf16", 24, 1, 2048)])
def test_host_buffer_slices_give_the_whole_calls_bits(dtype, n_q, n_kv, C):
    """Slices of 1 to 6 KV groups, grids with row blocks in parts among them, and a single KV head (unsliced)."""
    T = 1500
    gp = problem(14, n_q=n_q, n_kv=n_kv, T=T, C=C, n_retain=32, kv_budget=1100, dtype=dtype)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    want, want_k = gp.out.cpu(), gp.k.clone()
    host = [x.contiguous().pin_memory() for x in (gp.inp.q, gp.inp.k[:, :, T:T + C], gp.inp.v[:, :, T:T + C])]
    out_host = torch.zeros_like(host[0]).pin_memory()
    gp.k[:, :, T:] = 0
    gp.v[:, :, T:] = 0
    api.quoka_prefill_chunk_host(gp.p, gp.inp.ctx_len.clone(), *host, out_host, torch.zeros_like(gp.q), gp.k, gp.v, gp.out, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(out_host, want) and torch.equal(gp.k, want_k)


@pytest.mark.parametrize("n_q,n_kv,sliced", [(8, 2, True), (8, 4, True), (8, 8, True), (9, 3, True), (7, 1, False)])
def test_host_buffer_slices_of_a_grid_just_below_a_wave(n_q, n_kv, sliced):
    """128 to 144 row blocks that are not cut into parts: still copied in and out slice by slice (more launches than the
    device call's), with its bits."""
    C, T = 4096 if n_q < 9 else 4000, 3000
    gp = problem(16, n_q=n_q, n_kv=n_kv, T=T, C=C if n_q > 7 else 4700, n_retain=32, kv_budget=700)
    C = gp.C
    n0 = api.quoka_launch_count()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    n1 = api.quoka_launch_count()
    want = gp.out.cpu()
    host = [x.contiguous().pin_memory() for x in (gp.inp.q, gp.inp.k[:, :, T:T + C], gp.inp.v[:, :, T:T + C])]
    out_host = torch.zeros_like(host[0]).pin_memory()
    api.quoka_prefill_chunk_host(gp.p, gp.inp.ctx_len.clone(), *host, out_host, torch.zeros_like(gp.q), gp.k, gp.v, gp.out, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(out_host, want) and (api.quoka_launch_count() - n1 >= 2 * (n1 - n0)) == sliced


def test_a_host_buffer_call_that_is_refused_puts_nothing_on_any_stream():
    """The tensor-core kernels asked for, and more retained queries than they take: refused before the first copy, so that
    neither copies of it are in flight nor side streams forked in a capture."""
    T, C = 2000, 2048
    gp = problem(15, n_q=32, n_kv=8, T=T, C=C, n_retain=600, kv_budget=500, impl=api.IMPL_TENSOR)
    host = [x.contiguous().pin_memory() for x in (gp.inp.q, gp.inp.k[:, :, T:T + C], gp.inp.v[:, :, T:T + C])]
    out_host, q_dev, before = torch.zeros_like(host[0]).pin_memory(), torch.zeros_like(gp.q), api.quoka_launch_count()

    def call():
        with pytest.raises(api.QuokaError) as e:
            api.quoka_prefill_chunk_host(gp.p, gp.inp.ctx_len.clone(), *host, out_host, q_dev, gp.k, gp.v, gp.out, gp.ws)
        assert e.value.status == api.ERR_UNSUPPORTED

    call()
    torch.cuda.synchronize()
    assert not q_dev.any() and api.quoka_launch_count() == before
    with pytest.raises(api.QuokaError):
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    assert api.quoka_launch_count() == before
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        q_dev.add_(0)
        call()
    g.replay()
    torch.cuda.synchronize()
    assert not q_dev.any()


def test_host_buffer_entry_point_replayed_from_a_cuda_graph():
    # the sliced call forks to the library's two copy streams and joins again: captured as one graph and replayed
    shape = dict(n_q=32, n_kv=8, T=3000, C=2048, n_retain=64, kv_budget=700)
    gp = problem(12, **shape)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    want = gp.out.clone()
    T, C = shape["T"], shape["C"]
    q_host = gp.inp.q.contiguous().pin_memory()
    k_new = gp.inp.k[:, :, T:T + C].contiguous().pin_memory()
    v_new = gp.inp.v[:, :, T:T + C].contiguous().pin_memory()
    out_host = torch.zeros_like(q_host).pin_memory()
    q_dev = torch.zeros_like(gp.q)
    ctx_host = gp.inp.ctx_len.clone()

    def run():
        api.quoka_prefill_chunk_host(gp.p, ctx_host, q_host, k_new, v_new, out_host, q_dev, gp.k, gp.v, gp.out, gp.ws)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        run()                      # first use makes the copy streams: before any capture
        side.synchronize()
        with torch.cuda.graph(g, stream=side):
            run()
    torch.cuda.synchronize()
    for _ in range(2):
        out_host.zero_()
        gp.out.zero_()
        q_dev.zero_()
        gp.k[:, :, T:T + C].zero_()
        gp.v[:, :, T:T + C].zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out_host, want.cpu())
    assert api.quoka_last_device_status(gp.ws) == 0


# ---------------------------------------------------------------- selection step alone: exact integer parity
@pytest.mark.parametrize("T,B", [(5000, 600), (1024, 1), (1025, 1024), (33, 7), (70000, 8400)])
def test_select_keys_exact_with_planted_ties(T, B):
    r = np.random.default_rng(T)
    s = r.normal(size=(3, T)).astype(np.float32)
    s[0, :] = np.round(s[0] * 4) / 4            # heavy duplication: many ties at the threshold
    s[1, ::3] = 0.5
    s[1, 5] = -0.0
    s[1, 6] = 0.0
    inp = synth.make_chunk_inputs(0, 1, 3, 3, 64, T, 8, "bf16")
    gp = GpuProblem(inp, 4, kv_budget=B)
    gp.scores[0, :, :T] = torch.from_numpy(s).cuda()
    api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    want = O.select_keys(s.astype(np.float64), B)
    np.testing.assert_array_equal(gp.k_idx[0, :, :B].cpu().numpy(), want)
    assert int(gp.k_cnt[0]) == B


def scores_only_problem(T, B, n_kv=3):
    """Parameters and buffers for calling the selection step alone on rows of T scores: the caches are never
    touched by it, so they are a few rows long and only the declared sizes are large."""
    inp = synth.make_chunk_inputs(0, 1, n_kv, n_kv, 64, 8, 8, "bf16")
    gp = GpuProblem(inp, 4, kv_budget=B)
    gp.ctx_len.fill_(T)
    gp.p.max_ctx_len = T
    gp.p.kv_rows = T + 8
    gp.cap = api.quoka_kv_budget_cap(gp.p)
    gp.ws = api.alloc_workspace(gp.p)
    gp.scores = torch.zeros((1, n_kv, T), dtype=torch.float32, device="cuda")
    gp.k_idx = torch.full((1, n_kv, gp.cap), -7, dtype=torch.int32, device="cuda")
    return gp


@pytest.mark.parametrize("T,B", [(200000, 24000), (262144, 131072), (300000, 36000), (300000, 1)])
def test_select_keys_long_rows_exact_with_planted_ties(T, B):
    """Rows beyond 128K scores take the 8-CTA cluster of the register kernel (up to 256K) and, beyond that, the
    kernel that re-reads the scores in every digit pass."""
    r = np.random.default_rng(T + B)
    s = (r.normal(size=(3, T)) * 0.1).astype(np.float32)
    s[0, :] = np.round(s[0] * 64) / 64          # heavy duplication: many ties at the threshold
    s[1, ::5] = 0.05
    s[1, 5], s[1, 6] = -0.0, 0.0
    s[2, T - 1] = 3.0                           # the last row is the largest
    gp = scores_only_problem(T, B)
    gp.scores[0] = torch.from_numpy(s).cuda()
    api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    want = O.select_keys(s.astype(np.float64), B)
    np.testing.assert_array_equal(gp.k_idx[0, :, :B].cpu().numpy(), want)
    assert int(gp.k_cnt[0]) == B


@pytest.mark.parametrize("T,B", [(4097, 500), (31000, 3720), (40000, 39999)])
def test_select_keys_constant_and_narrow_rows(T, B):
    """Rows whose codes span almost nothing (the digits are taken relative to the row's smallest code): a
    constant row, a row of adjacent floats, a row with one outlier above a constant."""
    s = np.empty((3, T), dtype=np.float32)
    s[0, :] = 0.3125                                             # every score ties: the first B positions win
    base = np.float32(0.4)
    s[1, :] = base
    steps = np.random.default_rng(T).integers(0, 6, T)           # 0..5 ulps above the base, many ties per value
    for k in range(1, 6):
        v = base
        for _ in range(k):
            v = np.nextafter(v, np.float32(1.0))
        s[1, steps == k] = v
    s[2, :] = -0.75
    s[2, T // 2] = 0.9
    inp = synth.make_chunk_inputs(0, 1, 3, 3, 64, T, 8, "bf16")
    gp = GpuProblem(inp, 4, kv_budget=B)
    gp.scores[0, :, :T] = torch.from_numpy(s).cuda()
    api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    want = O.select_keys(s.astype(np.float64), B)
    np.testing.assert_array_equal(gp.k_idx[0, :, :B].cpu().numpy(), want)


def largest_by_order_code(s, B):
    """The B largest scores of each row by the kernels' order of floats: NaN above +inf (below -inf with the sign bit set),
    -0 equal to +0, equal codes by position; ascending positions."""
    u = s.view(np.uint32)
    u = np.where((u << 1) == 0, 0, u).astype(np.uint32)
    code = np.where(u >> 31, ~u, u | np.uint32(0x80000000)).astype(np.int64)
    return np.sort(np.argsort(-code, axis=1, kind="stable")[:, :B], axis=1)


@pytest.mark.parametrize("mode", ["cosine", "dot"])
@pytest.mark.parametrize("T,B,n_kv", [(700, 100, 6), (5000, 600, 6), (20011, 3000, 6), (20011, 3000, 33), (40000, 39000, 14)])
def test_select_keys_lists_b_rows_whatever_the_scores_are(T, B, n_kv, mode):
    """NaN and infinite scores, alone and beside ties at the threshold: still exactly B rows, in the kernels' order."""
    r = np.random.default_rng(T + B)
    s = (0.2 * r.normal(size=(n_kv, T))).astype(np.float32)
    s[0, :] = np.nan
    s[1, :] = np.where(r.random(T) < 0.7, np.float32(0.25), s[1])           # ties at the threshold, with some NaN above it
    s[1, r.permutation(T)[: B // 3]] = np.nan
    s[2, r.permutation(T)[: B + 7]] = np.nan                                # the threshold lies among the NaN
    s[3, r.permutation(T)[: T - B // 2]] = np.uint32(0xFFC00000).view(np.float32)     # among the NaN with the sign bit
    s[4, r.permutation(T)[: B // 2]] = np.inf
    s[4, r.permutation(T)[: T // 2]] = -np.inf
    s[5, 11] = np.nan
    gp = scores_only_problem(T, B, n_kv)
    gp.p.score_mode = {"cosine": api.SCORE_COSINE, "dot": api.SCORE_DOT}[mode]
    gp.scores[0] = torch.from_numpy(s).cuda()
    api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(gp.k_idx[0, :, :B].cpu().numpy(), largest_by_order_code(s, B))


@pytest.mark.parametrize("T,B,n_kv", [(600, 71, 33), (9001, 1080, 15), (33000, 3960, 8), (33000, 3960, 80), (140000, 16800, 5)])
def test_select_keys_of_rows_in_a_narrow_band(T, B, n_kv):
    """More rows in the threshold's bin than are ranked against each other: bands of a few codes and of many (one, two and
    three histograms over the codes), with a far-off row that widens the range.  Integer parity with the oracle."""
    r = np.random.default_rng(T)
    s = (0.25 + 1e-3 * r.normal(size=(n_kv, T))).astype(np.float32)
    s[1] = np.float32(0.25) + r.integers(0, 9000, T).astype(np.float32) * np.float32(2.0 ** -25)
    s[2] = (0.25 + 1e-4 * r.normal(size=T)).astype(np.float32)
    s[2, T // 3], s[2, T // 2] = -1.0, 1.0
    s[3, ::2] = np.float32(0.2505)
    gp = scores_only_problem(T, B, n_kv)
    gp.scores[0] = torch.from_numpy(s).cuda()
    api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(gp.k_idx[0, :, :B].cpu().numpy(), O.select_keys(s.astype(np.float64), B))


def test_select_keys_crowded_rows_are_not_far_slower_than_spread_ones():
    """8 rows of 32768 scores: equal ones, or ones in a narrow band, may cost a few more passes over the row (6.7 us spread,
    10 and 14 us crowded, back to back), not the 130 us of reading every CTA's histogram from every CTA."""
    gp = scores_only_problem(32768, 3932, 8)
    z = torch.randn(8, 32768, device="cuda", generator=torch.Generator("cuda").manual_seed(0))

    def best_us(scores):
        gp.scores[0] = scores
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 50)
        return min(times)

    spread = best_us(0.25 + 0.06 * z)
    assert best_us(torch.full_like(z, 0.25)) < 5 * spread and best_us(0.25 + 1e-3 * z) < 5 * spread


@pytest.mark.parametrize("C,dtype", [(1, "bf16"), (1, "f32"), (40, "f32")])
def test_queries_that_are_nan_leave_the_other_sequence_alone(C, dtype):
    """One sequence's queries are NaN (all its scores too): its list is still one of valid rows, and the other sequence's
    results are what they are without it."""
    gp = problem(77, batch=2, n_q=8, n_kv=2, T=[5000, 4100], C=C, dtype=dtype, n_retain=64, kv_budget=300)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    want = gp.out.clone()
    gp.q[0] = float("nan")
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert api.quoka_last_device_status(gp.ws) == 0
    assert (gp.k_idx[0].diff(dim=1) > 0).all() and gp.k_idx[0].min() >= 0 and gp.k_idx[0].max() < 5000
    assert torch.equal(gp.out[1], want[1]) and torch.isnan(gp.out[0].float()).all()


@pytest.mark.parametrize("d,dtype", [(128, "bf16"), (64, "bf16"), (128, "f32"), (64, "f32")])
@pytest.mark.parametrize("n_q,n_kv,T,B", [
    (4, 4, 1, 5),              # one cached row, a head per KV group
    (4, 2, 64, 63),            # 64 keys with the query's own: exactly one trip of one CTA
    (6, 2, 400, 127),          # groups of 3: a CTA of 4 heads with one unused; 128 keys
    (10, 2, 3000, 600),        # groups of 5: two CTAs per group; 8 parts, several trips
    (32, 2, 9000, 8300),       # groups of 16, a list beyond 8192 rows
])
def test_decode_attention_parts_and_groups(n_q, n_kv, T, B, d, dtype):
    """The generation step's attention at the edges of its parts, trips and head groups, with a list and without."""
    gp = problem(980 + T, batch=2, n_q=n_q, n_kv=n_kv, d=d, T=[T, max(1, T // 3)], C=1, dtype=dtype, n_retain=4, kv_budget=B)
    gp.run_staged()
    check_chain(gp)
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    for s in range(2):
        q, k, v, T_s = gp.oracle_inputs(s)
        dense, lse = O.dense_chunk_attention(q, k, v, T_s)
        check_attention(f64(gp.out[s]), dense, dtype)
        assert np.abs(f64(gp.lse[s]) - lse).max() <= 2e-3


@pytest.mark.parametrize("d,dtype", [(128, "bf16"), (64, "bf16"), (128, "f32"), (64, "f32")])
@pytest.mark.parametrize("n_q,n_kv", [(4, 4), (8, 2)])
def test_decode_attention_over_rows_whose_logits_overflow_to_minus_infinity(n_q, n_kv, d, dtype):
    """Whole trips of a warp, and every key of one part, may have logits of minus infinity: weights of zero, not NaN."""
    gp = problem(990 + d, n_q=n_q, n_kv=n_kv, d=d, T=400, C=1, dtype=dtype, n_retain=4, kv_budget=40)
    gp.q.abs_().add_(0.5)
    far = torch.cat([torch.arange(0, 140), torch.arange(200, 210)]).cuda()
    gp.k[:, :, far] = -3e38
    gp.k_idx[0] = torch.cat([far[:39], torch.tensor([399], device="cuda")]).int()
    gp.k_cnt.fill_(40)
    api.quoka_sparse_attn(gp.p, gp.q, gp.k, gp.v, gp.k_idx, gp.k_cnt, gp.out, gp.lse, gp.ws)
    listed, listed_lse = gp.out.clone(), gp.lse.clone()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v = f64(gp.q[0]), f64(gp.k[0]), f64(gp.v[0])
    want, lse = O.sparse_attention(q, k, v, 400, [gp.k_idx[0, h].cpu().numpy() for h in range(n_kv)])
    check_attention(f64(listed[0]), want, dtype)
    assert np.abs(f64(listed_lse[0]) - lse).max() <= 2e-3
    want, lse = O.dense_chunk_attention(q, k, v, 400)
    check_attention(f64(gp.out[0]), want, dtype)
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3


@pytest.mark.parametrize("listed", [False, True])
@pytest.mark.parametrize("group,d", [(1, 64), (4, 128)])
def test_f32_generation_step_keeps_the_thousands_of_small_weights(group, d, listed):
    """f32, one query, 16000 keys in one part (more KV groups than the GPU has room to cut): the first key of every lane's
    share has a weight e^17 times the others', of which a thousand and more follow, each below half an ulp of the lane's sum.
    Added one by one they all vanished (7e-4 of 16, times values of 3)."""
    b, n_kv, T = 19, 8, 16000
    first = torch.arange(8)[:, None] * (512 // d) + torch.arange(128 // d)
    g = torch.Generator("cuda").manual_seed(5)
    q = torch.zeros(b, n_kv * group, 1, d, device="cuda")
    q[..., 0] = d ** 0.5                                         # logits are the keys' first elements
    k = 0.1 * torch.randn(b, n_kv, T + 1, d, device="cuda", generator=g)
    k[:, :, first.flatten().cuda(), 0] = 17.0
    v = 3.0 + torch.rand(b, n_kv, T + 1, d, device="cuda", generator=g)
    v[:, :, first.flatten().cuda()] = -5.0
    out, lse = torch.empty_like(q), torch.empty(b, n_kv * group, 1, device="cuda")
    ctx = torch.full((b,), T, dtype=torch.int32, device="cuda")
    p = api.make_params(q, k, out, ctx, n_retain=4, kv_budget=T - 3, max_ctx_len=T)
    ws = api.alloc_workspace(p)
    if listed:
        idx = torch.arange(T - 3, dtype=torch.int32, device="cuda").expand(b, n_kv, T - 3).contiguous()
        api.quoka_sparse_attn(p, q, k, v, idx, torch.full_like(ctx, T - 3), out, lse, ws)
    else:
        api.quoka_dense_chunk_attn(p, q, k, v, out, lse, ws)
    torch.cuda.synchronize()
    rows = torch.cat([torch.arange(T - 3 if listed else T), torch.tensor([T])]).cuda()
    w = torch.exp(k[:, :, rows, 0].double())
    want = (w[:, :, None] @ v[:, :, rows].double())[:, :, 0] / w.sum(-1, keepdim=True)
    want = want.repeat_interleave(group, 1)
    assert (out[:, :, 0].double() - want).abs().max() <= 2e-5
    assert (lse[:, :, 0].double() - torch.log(w.sum(-1)).repeat_interleave(group, 1)).abs().max() <= 1e-5


@pytest.mark.parametrize("T,max_ctx", [(100, 4096), (100, 1000), (4000, 4096)])
def test_generation_step_over_a_callers_own_list(T, max_ctx):
    """A list in any order, with repeated rows, longer than the cache even: every entry counts."""
    inp = synth.make_chunk_inputs(78, 1, 8, 2, 128, T, 1, "bf16", capacity=max_ctx + 1)
    gp = GpuProblem(inp, 4, kv_budget=300, max_ctx_len=max_ctx)
    gp.k_idx.copy_(torch.randint(0, T, gp.k_idx.shape, generator=torch.Generator().manual_seed(T)))
    gp.k_cnt.fill_(300)
    api.quoka_sparse_attn(gp.p, gp.q, gp.k, gp.v, gp.k_idx, gp.k_cnt, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v, _ = gp.oracle_inputs(0)
    want, lse = O.sparse_attention(q, k, v, T, [gp.k_idx[0, h].cpu().numpy() for h in range(2)])
    check_attention(f64(gp.out[0]), want, "bf16")
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_generation_step_over_an_infinite_value(dtype):
    """An infinite value among hundreds makes its output infinite, not NaN, and no other."""
    gp = problem(79, n_q=4, n_kv=2, d=64, T=900, C=1, dtype=dtype, n_retain=4, kv_budget=900)
    gp.v[:, 0, 5, 7], gp.v[:, 0, 600, 9] = float("inf"), float("-inf")
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert (gp.out[0, :2, 0, 7] == float("inf")).all() and (gp.out[0, :2, 0, 9] == float("-inf")).all()
    assert int(torch.isfinite(gp.out).sum()) == gp.out.numel() - 4


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("T,max_ctx,B,n_q,n_kv,d,dtype", [
    ([2049], 2049, 64, 8, 2, 128, "bf16"),        # just beyond the two-launch form: 258 positions per CTA
    ([0, 5, 4096], 4096, 200, 6, 2, 64, "f32"),   # an empty cache, a budget that covers one, exactly 512 positions per CTA
    ([4097, 300], 9000, 299, 8, 4, 128, "f32"),   # two items per thread, the second CTA's last rows alone
    ([33000], 33000, 3000, 5, 1, 64, "bf16"),     # beyond eight items per thread; two head blocks per group
    ([40000], 70000, 8448, 3, 3, 128, "bf16"),    # as many listed rows as a CTA can keep
])
def test_decode_select_and_attend_in_one_launch(T, max_ctx, B, n_q, n_kv, d, dtype, paged):
    """The generation step's selection + attention kernel: its list and its output against the staged calls (same bits),
    those against the oracle; then with every listed row in the first CTAs' parts of the cache, at equal scores."""
    inp = synth.make_chunk_inputs(1010 + d, len(T), n_q, n_kv, d, T, 1, dtype, capacity=max_ctx + 1)
    if paged:
        inp = synth.to_paged(inp, 3)
        extra = -(-(max_ctx + 1) // 64) - inp.block_table.shape[1]
        inp.block_table = torch.nn.functional.pad(inp.block_table, (0, max(extra, 0)), value=-1)
    gp = GpuProblem(inp, 4, kv_budget=B, paged=paged, max_ctx_len=max_ctx)
    for _ in range(2):
        gp.run_staged()
        check_chain(gp)
        want_out, want_idx, want_cnt = gp.out.clone(), gp.k_idx.clone(), gp.k_cnt.clone()
        gp.out.zero_(); gp.k_idx.fill_(-9); gp.k_cnt.fill_(-9)
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
        torch.cuda.synchronize()
        assert torch.equal(gp.out, want_out) and torch.equal(gp.k_idx, want_idx) and torch.equal(gp.k_cnt, want_cnt)
        gp.out.zero_()
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)      # no list asked for
        torch.cuda.synchronize()
        assert torch.equal(gp.out, want_out) and api.quoka_last_device_status(gp.ws) == 0
        if paged:
            break
        n = min(t for t in T if t > 0)
        n = min(n, B + 30)                          # equal keys along the group's queries: the cut lies among them
        toward = gp.q.view(len(T), n_kv, n_q // n_kv, d).float().mean(2)[:, :, None] + 0.5 * gp.k[:, :, :1].float()
        gp.k[:, :, :n] = toward.to(gp.k.dtype)      # (cosine well below 1: Q-bar's own rounding may exceed it by 2^-8)
        inp.k = gp.k.cpu()


@pytest.mark.parametrize("cached_norms,paged", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("d,dtype,group", [(128, "bf16", 4), (64, "bf16", 3), (128, "f32", 1), (64, "f32", 40)])
@pytest.mark.parametrize("T", [[1, 8, 15, 17], [0, 31, 0, 33], [3000, 63, 0, 1], [65] * 35])
def test_decode_scoring_units(T, d, dtype, group, cached_norms, paged):
    """The generation step's scoring kernel: lengths around its units of 8 to 32 rows, empty sequences between others,
    more than 32 sequences; and the fused call, which forms Q-bar inside it, against the staged calls."""
    gp = problem(990 + d, batch=len(T), n_q=2 * group, n_kv=2, d=d, T=T, C=1, dtype=dtype, n_retain=4, kv_budget=12,
                 paged=paged, cached_norms=cached_norms)
    gp.run_staged()
    check_chain(gp)
    want_out, want_idx = gp.out.clone(), gp.k_idx.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, want_out) and torch.equal(gp.k_idx, want_idx)


@pytest.mark.gpu
@pytest.mark.parametrize("n_q,n_kv,d,C,T,B,paged", [
    (32, 4, 64, 777, 6000, 1500, False),    # P in place, three S buffers; the last row block has one Q tile, of nine rows
    (32, 4, 64, 384, 3000, 2999, True),     # and of 128
    (32, 8, 128, 633, 6000, 1500, True),    # pairs: one S buffer, P apart
    (32, 32, 128, 640, 2500, 700, False),   # the same with one head per tile
])
def test_q_tiles_that_walk_many_key_tiles(n_q, n_kv, d, C, T, B, paged):
    """Row blocks of two Q tiles and of one over dozens of key tiles: the buffers of scores and weights go round many times.
    Sparse (staged, and the fused call five times with the same bits) and dense, against the oracle."""
    gp = problem(2000 + C, n_q=n_q, n_kv=n_kv, d=d, T=T, C=C, n_retain=32, kv_budget=B, paged=paged)
    gp.run_staged()
    check_chain(gp, attn_rows=200)
    staged = gp.out.clone()
    for _ in range(5):
        gp.out.zero_()
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
        torch.cuda.synchronize()
        assert torch.equal(gp.out, staged)
    q, k, v, _ = gp.oracle_inputs(0)
    heads, rows = stratified_rows(n_q, C, 200, 5)
    want = O.sparse_attention_rows(q, k, v, T, [np.arange(T)] * n_kv, heads, rows)
    for _ in range(2):
        gp.out.zero_()
        api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
        torch.cuda.synchronize()
        check_attention(f64(gp.out[0])[heads, rows], want, "bf16")
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("n_q,n_kv,C", [
    (4, 4, 129), (4, 4, 256),           # one tile in each CTA of a pair, the second one's of one row and full
    (4, 4, 257), (4, 4, 385),           # a third tile of one row, a fourth: the As begin two key tiles after the Bs
    (4, 4, 512), (4, 4, 700),           # full row blocks; a last one without Bs
    (4, 2, 64), (4, 2, 65), (4, 2, 193),
    (12, 4, 85), (12, 4, 169),          # 42 positions per tile
])
def test_rows_of_a_pair_of_ctas(n_q, n_kv, C):
    """Few query heads per KV head at head_dim 128, chunk lengths at the edges of a pair's tiles: sparse (staged and fused, the
    same bits) and dense, every row and its log-sum-exp against the oracle."""
    T = 1500
    gp = problem(2100 + C, n_q=n_q, n_kv=n_kv, T=T, C=C, n_retain=16, kv_budget=300)
    gp.run_staged()
    check_chain(gp, attn_rows=400)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    gp.out.zero_()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v, t = gp.oracle_inputs(0)
    dense, lse = O.dense_chunk_attention(q, k, v, t)
    check_attention(f64(gp.out[0]), dense, "bf16")
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.parametrize("n_q,n_kv,d,C,T,B", [
    (32, 8, 128, 1300, 9000, 5000),     # pairs, 11 row blocks: the lightest in parts after the whole ones, ragged last block
    (24, 8, 64, 1800, 7000, 6000),      # one-CTA kernel, 22 row blocks
    (32, 8, 128, 1281, 6000, 6000),     # the budget covers the cache: the list is the identity
])
def test_attention_with_its_lightest_row_blocks_in_parts(n_q, n_kv, d, C, T, B):
    """Grids of a full wave and a rest: whole row blocks and parts in one call, sparse (staged and fused) and dense, twice
    over the same workspace (the arrival counters go back to zero), every row against the oracle for two KV groups."""
    gp = problem(1000 + C, n_q=n_q, n_kv=n_kv, d=d, T=T, C=C, n_retain=32, kv_budget=B)
    assert n_q * -(-C // 256) > 148 and n_q * -(-C // 256) % 148
    gp.run_staged()
    check_chain(gp, attn_rows=200)
    staged = gp.out.clone()
    for _ in range(2):
        gp.out.zero_()
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
        torch.cuda.synchronize()
        assert torch.equal(gp.out, staged)
    q, k, v, _ = gp.oracle_inputs(0)
    for _ in range(2):
        gp.out.zero_()
        api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
        torch.cuda.synchronize()
        heads, rows = stratified_rows(n_q, C, 200, 5)
        want = O.sparse_attention_rows(q, k, v, T, [np.arange(T)] * n_kv, heads, rows)
        check_attention(f64(gp.out[0])[heads, rows], want, "bf16")


@pytest.mark.parametrize("n_q,n_kv,d,C,tail,T", [
    (32, 8, 128, 2048, 1500, 4096),       # no parts for the whole chunk, 12 MiB of them for the rest of the prompt
    (40, 8, 64, 2048, 1270, 8192),        # parts in both, more of them for the shorter chunk
    (80, 10, 64, 2048, 260, 8192),        # 160 blocks of 256 positions, 90 CTAs of packed heads
])
def test_a_workspace_made_for_the_longest_chunk_serves_the_shorter_ones(n_q, n_kv, d, C, tail, T):
    """The scratch of grids of a wave or more may be missing: what was sized for another chunk of the same prompt is accepted,
    the results are right, nothing behind the given bytes is touched; below the intermediates it is still refused."""
    gp = problem(1300 + tail, n_q=n_q, n_kv=n_kv, d=d, T=T, C=tail, n_retain=64, kv_budget=T // 8)
    full = GpuProblem(synth.make_chunk_inputs(0, 1, n_q, n_kv, d, 8, C, "bf16"), 64, kv_budget=T // 8)
    full.p.max_ctx_len, full.p.kv_rows = T, T + C
    n = api.quoka_workspace_size(full.p)
    assert n < gp.ws.numel()
    guarded = torch.full((n + (1 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
    guarded[:256] = 0
    ws, q, k, v = guarded[:n], *gp.oracle_inputs(0)[:3]
    heads, rows = stratified_rows(n_q, tail, 64, 5)
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, ws)
    torch.cuda.synchronize()
    idx = [gp.k_idx[0, h].cpu().numpy() for h in range(n_kv)]
    check_attention(f64(gp.out[0])[heads, rows], O.sparse_attention_rows(q, k, v, T, idx, heads, rows), "bf16")
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, None, ws)
    torch.cuda.synchronize()
    check_attention(f64(gp.out[0])[heads, rows], O.sparse_attention_rows(q, k, v, T, [np.arange(T)] * n_kv, heads, rows), "bf16")
    assert (guarded[n:] == 0x5A).all() and api.quoka_last_device_status(ws) == 0
    with pytest.raises(api.QuokaError) as e:
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, ws[:n_kv * T * 4])
    assert e.value.status == api.ERR_WORKSPACE


@pytest.mark.parametrize("n_q,n_kv,d,tail", [
    (32, 8, 128, 2), (32, 8, 128, 64), (32, 8, 128, 512), (32, 8, 128, 896), (32, 4, 64, 64), (32, 4, 64, 900), (32, 32, 128, 300),
])
def test_the_end_of_a_prompt_runs_in_the_workspace_of_its_longest_chunk(n_q, n_kv, d, tail):
    """A chunk far below a wave after chunks of 2048: accepted, and with the bits of a call that has its own workspace, that is
    in as many parts.  Without any room for parts it is accepted too, and right."""
    T, C = 32768, 2048
    gp = problem(1350 + tail, n_q=n_q, n_kv=n_kv, d=d, T=T, C=tail, n_retain=64, kv_budget=3932)
    full = GpuProblem(synth.make_chunk_inputs(0, 1, n_q, n_kv, d, 8, C, "bf16"), 64, kv_budget=3932)
    full.p.max_ctx_len, full.p.kv_rows = T, T + C
    plain = api.QuokaParams.from_buffer_copy(gp.p)
    plain.impl = api.IMPL_SIMT                                  # (no parts: the intermediates alone)
    heads, rows = stratified_rows(n_q, tail, 64, 5)
    q, k, v = gp.oracle_inputs(0)[:3]
    got = []
    for n in (gp.ws.numel(), api.quoka_workspace_size(full.p), api.quoka_workspace_size(plain)):
        guarded = torch.full((n + (1 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
        guarded[:256] = 0
        ws = guarded[:n]
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, ws)
        sparse = gp.out.clone()
        api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, None, ws)
        torch.cuda.synchronize()
        got.append((sparse, gp.out.clone()))
        assert (guarded[n:] == 0x5A).all() and api.quoka_last_device_status(ws) == 0
    assert torch.equal(got[1][0], got[0][0]) and torch.equal(got[1][1], got[0][1])
    idx = [gp.k_idx[0, h].cpu().numpy() for h in range(n_kv)]
    for sparse, dense in got[1:]:
        check_attention(f64(sparse[0])[heads, rows], O.sparse_attention_rows(q, k, v, T, idx, heads, rows), "bf16")
        check_attention(f64(dense[0])[heads, rows], O.sparse_attention_rows(q, k, v, T, [np.arange(T)] * n_kv, heads, rows), "bf16")


@pytest.mark.parametrize("n_q,n_kv,C,T,B", [
    (8, 2, 256, [4096], 2048),          # 4 clusters of eight CTAs
    (8, 4, 257, [2500, 40], 2000),      # a row block of one row; a list shorter than a tile: parts without a tile
    (32, 8, 130, [3000], 1500),         # 16 clusters of six
    (32, 8, 2, [1030], 1024),           # two query rows
    (32, 8, 400, [3000], 3000),         # two parts through memory, the list is the identity; dense: one CTA, whole
    (2, 1, 64, [1100], 1025),           # one cluster
])
def test_attention_parts_in_a_cluster(n_q, n_kv, C, T, B):
    """Short grids of the pair kernel, whose parts merge through distributed shared memory: sparse (staged and fused, the
    same bits) and dense, every row and its log-sum-exp against the oracle."""
    gp = problem(1100 + C, batch=len(T), n_q=n_q, n_kv=n_kv, T=T, C=C, n_retain=16, kv_budget=B)
    gp.run_staged()
    check_chain(gp, attn_rows=400)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    for s in range(gp.b):
        q, k, v, t = gp.oracle_inputs(s)
        dense, lse = O.dense_chunk_attention(q, k, v, t)
        check_attention(f64(gp.out[s]), dense, "bf16")
        assert np.abs(f64(gp.lse[s]) - lse).max() <= 2e-3


# n_q, n_kv, C, T, B, call; kernel, CTAs of a cluster, grid of its launch on 148 SMs
FORMS = [
    (16, 16, 1030, 600, 300, "dense", "attn_tc", 1, (16, 9, 1)),         # one CTA, one Q tile, whole; the last one of six rows
    (16, 16, 1030, 600, 300, "sparse", "attn_tc", 1, (16, 9, 1)),
    (8, 8, 1030, 3000, 1500, "dense", "attn_tc", 1, (8, 18, 1)),         # in two parts
    (128, 128, 200, 600, 300, "sparse", "attn_tc", 1, (128, 1, 1)),      # two Q tiles, whole
    (32, 32, 200, 8000, 6000, "sparse", "attn_tc", 1, (32, 4, 1)),       # in four parts
    (37, 1, 40, 3000, 3000, "sparse", "attn_tc", 1, (37, 4, 1)),         # the list is the identity
    (32, 32, 100, 3000, 1500, "dense", "attn_tc", 1, (32, 4, 1)),
    (74, 2, 64, 1000, 120, "dense", "attn_tc", 1, (74, 1, 1)),           # a pair's second CTA would be idle
    (32, 32, 633, 1500, 700, "sparse", "attn_tc_pair", 2, (64, 2, 1)),   # pairs, two Q tiles each, whole
    (4, 4, 64, 1500, 700, "sparse", "attn_tc_pair", 2, (8, 1, 1)),       # one
    (32, 8, 400, 3000, 3000, "sparse", "attn_tc_pair", 2, (16, 8, 1)),   # two parts through memory
    (24, 24, 40, 3000, 1500, "sparse", "attn_tc_pair", 4, (48, 2, 1)),   # 24 clusters of four, one Q tile
    (24, 24, 64, 1500, 700, "dense", "attn_tc_pair", 4, (48, 2, 1)),
    (32, 8, 257, 3000, 3000, "sparse", "attn_tc_pair", 4, (16, 6, 1)),   # and two
    (32, 8, 300, 3000, 1500, "dense", "attn_tc_pair", 4, (16, 6, 1)),
    (8, 8, 257, 3000, 1500, "sparse", "attn_tc_pair", 6, (16, 6, 1)),    # 16 clusters of six
    (8, 8, 300, 3000, 3000, "sparse", "attn_tc_pair", 8, (16, 4, 1)),    # 8 of eight
]


@pytest.mark.gpu
def test_attention_forms_are_the_ones_meant():
    """The launches of the calls in FORMS, by the library's launch log."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the plan goes by the number of SMs")
    code = """
import sys, torch
from paper_2602_08722_b200 import api
from tests.test_gpu_parity import FORMS
for n_q, n_kv, C, T, B, call, *_ in FORMS:
    q = torch.zeros(1, n_q, C, 128, dtype=torch.bfloat16, device="cuda")
    k = torch.zeros(1, n_kv, T + C, 128, dtype=torch.bfloat16, device="cuda")
    p = api.make_params(q, k, q.clone(), torch.full((1,), T, dtype=torch.int32, device="cuda"), n_retain=16, kv_budget=B, max_ctx_len=T)
    ws, out = api.alloc_workspace(p), torch.empty_like(q)
    print("form", file=sys.stderr, flush=True)
    if call == "dense":
        api.quoka_dense_chunk_attn(p, q, k, k, out, None, ws)
    else:
        api.quoka_prefill_chunk(p, q, k, k, out, None, None, ws)
    torch.cuda.synchronize()
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", code], cwd=root, env=dict(os.environ, QUOKA_LOG="1"), capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr[-2000:]
    logs = run.stderr.split("form\n")[1:]
    assert len(logs) == len(FORMS)
    for form, log in zip(FORMS, logs):
        got = re.findall(r"\] (attn\w+) +grid \((\d+),(\d+),(\d+)\).* cluster (\d+)", log)
        assert [(g[0], int(g[4]), (int(g[1]), int(g[2]), int(g[3]))) for g in got] == [form[6:]], (form, log)


@pytest.mark.gpu
@pytest.mark.parametrize("n_q,n_kv,C,T,B,call", [f[:6] for f in FORMS])
def test_attention_forms(n_q, n_kv, C, T, B, call):
    """Every form of row block and of parts at head_dim 128: two calls over one workspace with the same bits, against the oracle."""
    gp = problem(2200 + C, n_q=n_q, n_kv=n_kv, T=T, C=C, n_retain=16, kv_budget=B)
    heads, rows = stratified_rows(n_q, C, 400, 5)
    if call == "sparse":
        gp.run_staged()
        check_chain(gp, attn_rows=400)
    got = gp.out.clone()
    for rep in range(2):
        gp.out.zero_()
        if call == "sparse":
            api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
        else:
            api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
        torch.cuda.synchronize()
        if call == "dense" and rep == 0:
            q, k, v, t = gp.oracle_inputs(0)
            want = O.sparse_attention_rows(q, k, v, t, [np.arange(t)] * n_kv, heads, rows)
            check_attention(f64(gp.out[0])[heads, rows], want, "bf16")
            got = gp.out.clone()
        assert torch.equal(gp.out, got)
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n_q,n_kv,C", [
    (32, 2, 70), (32, 2, 301),          # 16 heads to a tile, 8 positions
    (26, 1, 40), (26, 2, 300),          # 26: 4 positions and 24 rows left over, or 13: 9 and 11
    (64, 2, 33), (40, 1, 130),          # 32; 20 or 8
    (37, 1, 20), (37, 1, 200),          # a prime above 32: one head to a tile
    (19, 1, 90), (28, 1, 610),          # one or 19; 14, 7 or 4
])
def test_many_heads_per_kv_head(n_q, n_kv, C, d):
    """Groups of 13 to 40 heads: sparse (staged and fused, the same bits) and dense, sampled rows against the oracle."""
    T = 2300
    gp = problem(2300 + C, n_q=n_q, n_kv=n_kv, d=d, T=T, C=C, n_retain=24, kv_budget=900)
    gp.run_staged()
    check_chain(gp, attn_rows=300)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    gp.out.zero_()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v, t = gp.oracle_inputs(0)
    heads, rows = stratified_rows(n_q, C, 300, 5)
    want = O.sparse_attention_rows(q, k, v, t, [np.arange(t)] * n_kv, heads, rows)
    check_attention(f64(gp.out[0])[heads, rows], want, "bf16")
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
def test_a_dense_chunk_of_more_row_blocks_than_a_grid_dimension_holds():
    """32 heads to a tile would make 65537 row blocks of 8 positions: sampled rows against a softmax in 64 bits."""
    C, n_q, d = 65536 * 8 + 3, 32, 64
    g = torch.Generator("cuda").manual_seed(3)
    q = torch.randn(1, n_q, C, d, dtype=torch.bfloat16, device="cuda", generator=g)
    k, v = (torch.randn(1, 1, C, d, dtype=torch.bfloat16, device="cuda", generator=g) for _ in range(2))
    out, ctx = torch.zeros_like(q), torch.zeros(1, dtype=torch.int32, device="cuda")
    p = api.make_params(q, k, out, ctx, n_retain=C, kv_budget=64, max_ctx_len=0)
    ws = api.alloc_workspace(p)
    api.quoka_dense_chunk_attn(p, q, k, v, out, None, ws)
    torch.cuda.synchronize()
    assert api.quoka_last_device_status(ws) == 0
    for h, r in ((0, 0), (31, 200), (5, 70001), (17, C // 2), (0, C - 4), (31, C - 3), (9, C - 1)):
        w = torch.softmax(k[0, 0, :r + 1].double() @ q[0, h, r].double() / d ** 0.5, 0)
        want = (w[:, None] * v[0, 0, :r + 1].double()).sum(0)
        check_attention(f64(out[0, h, r])[None], f64(want)[None], "bf16")


@pytest.mark.parametrize("n_q,C,n_retain,d,dtype", [
    (4, 2, 1, 128, "bf16"),             # one row per CTA
    (4, 65, 64, 64, "f32"),             # 33 rows: a block of one row
    (4, 500, 200, 128, "bf16"),         # clusters of eight, 63 rows
    (4, 1025, 130, 64, "bf16"),         # clusters of eight with a short last slice
    (4, 2047, 300, 128, "f32"),         # 256 rows, more than shared memory keeps; still counted
    (4, 2049, 40, 128, "bf16"),         # 257 rows: sorted in runs
    (4, 4099, 513, 128, "bf16"),        # 513 rows, kept in part
    (80, 510, 200, 128, "bf16"),        # several waves: two CTAs of 255 rows, the last block not full
    (80, 1023, 64, 128, "f32"),         # and of 512, kept in part
])
def test_query_ranks_at_the_edges_of_a_slice(n_q, C, n_retain, d, dtype):
    """Slices that are counted, sorted, kept in part: the ranks of random rows against the oracle, and of rows that have one
    of two values (equal cosines go by position) exactly."""
    gp = problem(1200 + C, n_q=n_q, n_kv=2, d=d, T=40, C=C, dtype=dtype, n_retain=n_retain, kv_budget=8)
    api.quoka_select_queries(gp.p, gp.q, gp.q_idx, gp.qbar, gp.ws)
    torch.cuda.synchronize()
    _, cos = O.select_queries(f64(gp.q[0]), n_retain)
    check_query_ranks(gp.q_idx[0].cpu().numpy(), cos, n_retain)
    pick = np.random.default_rng(C).random(C) < 0.3
    q2 = gp.q[:, :, :1].expand_as(gp.q).clone()
    q2[:, :, torch.from_numpy(np.nonzero(pick)[0]).cuda()] = -gp.q[:, :, 1:2]
    api.quoka_select_queries(gp.p, q2, gp.q_idx, gp.qbar, gp.ws)
    torch.cuda.synchronize()
    mean = f64(q2[0]).mean(axis=1)
    for h in range(n_q):
        c = f64(q2[0, h]) @ mean[h] / np.linalg.norm(f64(q2[0, h]), axis=1)
        low = c < 0.5 * (c.min() + c.max())
        want = np.concatenate([np.nonzero(low)[0], np.nonzero(~low)[0]])[:n_retain] if pick.any() and not pick.all() else np.arange(n_retain)
        assert np.array_equal(gp.q_idx[0, h].cpu().numpy(), want)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("T,C,B,n_q,n_kv,d,n_retain", [
    (63, 2, 40, 4, 2, 128, 1),          # fewer keys than a tile, two query rows
    (129, 63, 128, 2, 1, 64, 16),       # the last tile of the list holds one key
    (2000, 65, 700, 3, 3, 128, 33),     # parts of unequal length, a row block of one row, 33 retained queries
    (1500, 640, 64, 32, 8, 64, 32),     # more row blocks than SMs: one part
])
def test_f32_tiles_at_their_edges(T, C, B, n_q, n_kv, d, n_retain, paged):
    """The f32 kernels at the edges of their 64 x 64 tiles and of the parts a row block's keys are cut into."""
    gp = problem(970 + T, n_q=n_q, n_kv=n_kv, d=d, T=T, C=C, dtype="f32", n_retain=n_retain, kv_budget=B, paged=paged)
    gp.run_staged()
    check_chain(gp)
    q, k, v, _ = gp.oracle_inputs(0)
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    dense, lse = O.dense_chunk_attention(q, k, v, T)
    check_attention(f64(gp.out[0]), dense, "f32")
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3


def test_f32_scoring_of_few_queries_is_not_slower_than_of_a_full_block():
    """2 retained queries against 32 (20 us each at this size; 58 us for 2 while a block repeated its last row)."""
    best = {}
    for n in (2, 32):
        gp = problem(31, n_q=2, n_kv=2, d=64, T=32768, C=n, dtype="f32", n_retain=64, kv_budget=64)
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                api.quoka_score_keys(gp.p, gp.qbar, gp.k, gp.scores, gp.ws)
            b.record()
            torch.cuda.synchronize()
            best[n] = min(best.get(n, 1e9), a.elapsed_time(b))
    assert best[2] < 1.5 * best[32]


@pytest.mark.parametrize("d,C", [(128, 70), (64, 70), (128, 1)])
def test_f32_products_beyond_the_range_of_logits_within_it(d, C):
    """q . k overflows, q . k / sqrt(d) does not: the row is one-hot, not NaN."""
    gp = problem(83, n_q=4, n_kv=2, d=d, T=300, C=C, dtype="f32", n_retain=8, kv_budget=60)
    gp.q[0, 1, C // 2] = 0
    gp.q[0, 1, C // 2, 5] = 2e38
    gp.inp.q = gp.q.cpu()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v, T = gp.oracle_inputs(0)
    check_attention(f64(gp.out[0]), O.dense_chunk_attention(q, k, v, T)[0], "f32")
    assert torch.isfinite(gp.lse).all()


@pytest.mark.parametrize("d,C,T,bound", [(128, 192, 4096, 2.5e-7), (64, 600, 3000, 2.3e-7)])
def test_f32_attention_against_64_bits(d, C, T, bound):
    """Relative error (2-norm) of the f32 attention: 2.3e-7 and 2.1e-7 here, the rounding of sums of 128 products and of a few
    hundred weights; 2.7e-7 and 2.5e-7 with longer chains and the last sums in 32 bits, 2.0e-7 and 1.9e-7 in the scalar kernel."""
    g = torch.Generator("cuda").manual_seed(0)
    q = torch.randn(1, 4, C, d, device="cuda", generator=g) + torch.randn(1, 4, 1, d, device="cuda", generator=g)
    k, v = (torch.randn(1, 2, T + C, d, device="cuda", generator=g) for _ in range(2))
    out, ctx = torch.empty_like(q), torch.full((1,), T, dtype=torch.int32, device="cuda")
    p = api.make_params(q, k, out, ctx, n_retain=16, kv_budget=64, max_ctx_len=T)
    api.quoka_dense_chunk_attn(p, q, k, v, out, None, api.alloc_workspace(p))
    logits = q.double() @ k.double().repeat_interleave(2, 1).transpose(-1, -2) / d ** 0.5
    logits[..., T:].masked_fill_(torch.triu(torch.ones(C, C, device="cuda", dtype=torch.bool), 1), float("-inf"))
    want = torch.softmax(logits, -1) @ v.double().repeat_interleave(2, 1)
    assert (out.double() - want).norm() <= bound * want.norm()


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("T,C,B,n_q,n_kv,d", [(2000, 200, 300, 4, 2, 128), (100, 64, 30, 2, 1, 64), (700, 650, 100, 32, 8, 64)])
def test_f32_values_of_later_rows_do_not_reach_earlier_ones(T, C, B, n_q, n_kv, d, bad):
    """A value that is not finite reaches the rows that attend it and no others, although a tile holds both."""
    gp = problem(960 + T, n_q=n_q, n_kv=n_kv, d=d, T=T, C=C, dtype="f32", n_retain=16, kv_budget=B)
    for call in ("sparse", "dense"):
        got = []
        for row in (None, C // 2 + 3):
            if row is not None:
                gp.v[:, :, T + row, d // 3] = bad
            if call == "sparse":
                api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
            else:
                api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, None, gp.ws)
            torch.cuda.synchronize()
            got.append(gp.out.clone())
        gp.v[:, :, T + row, d // 3] = 0.5
        assert torch.isfinite(got[0]).all()
        assert torch.equal(got[1][:, :, :row], got[0][:, :, :row])
        assert not torch.isfinite(got[1][:, :, row:, d // 3]).any()


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("T,C,B,n_q,n_kv,d", [
    (3000, 700, 1500, 4, 4, 128),       # row blocks of up to four key tiles: pairs in clusters
    (3000, 400, 3000, 32, 8, 128),      # pairs in parts through memory; dense: one CTA, whole
    (3000, 1030, 1500, 8, 8, 128),      # dense: one CTA in parts through memory
    (1500, 900, 200, 16, 16, 128),      # whole pairs
    (2500, 600, 2300, 8, 8, 64),        # head_dim 64: parts
    (700, 1300, 100, 16, 16, 64),       # and whole
])
def test_bf16_values_of_later_tiles_do_not_reach_earlier_rows(T, C, B, n_q, n_kv, d, bad):
    """A value that is not finite leaves the bits of all rows that end in an earlier key tile (a tile that a row does not see
    adds 0 * inf to it until its first own tile wipes the sum), and reaches the rows that attend it."""
    gp = problem(970 + T, n_q=n_q, n_kv=n_kv, d=d, T=T, C=C, n_retain=16, kv_budget=B)
    row = C // 2 + 77
    for call in ("sparse", "dense"):
        got = []
        for broken in (False, True):
            keep = gp.v[:, :, T + row, d // 3].clone()
            if broken:
                gp.v[:, :, T + row, d // 3] = bad
            if call == "sparse":
                api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
            else:
                api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, None, gp.ws)
            torch.cuda.synchronize()
            got.append(gp.out.clone())
            gp.v[:, :, T + row, d // 3] = keep
        first = T if call == "dense" else 0                      # where a tile of the walk begins
        end = (first + row) // 128 * 128 - first
        assert end > 0 and torch.isfinite(got[0]).all()
        assert torch.equal(got[1][:, :, :end], got[0][:, :, :end])
        assert not torch.isfinite(got[1][:, :, row:, d // 3]).any()


@pytest.mark.parametrize("mode", ["cosine", "dot"])
@pytest.mark.parametrize("T,n_kv", [(513, 3), (8193, 8), (16385, 8), (16385, 33), (20011, 73), (32768, 14), (32769, 15)])
def test_select_keys_every_cluster_width(T, n_kv, mode):
    """Rows cut into 1 / 2 / 4 / 8 CTAs (by length and number of rows): a spread row, rows whose threshold falls into a
    bin of more rows than are ranked against each other (equal and nearly equal scores, with the cut inside a CTA and
    at a CTA's edge), scores outside [-1, 1] and rows of two values.  Integer parity with the oracle."""
    B = T // 7 + 1
    r = np.random.default_rng(T + n_kv)
    s = (0.25 + 0.03 * r.normal(size=(n_kv, T))).astype(np.float32)
    s[0, :] = np.float32(0.3) + r.integers(0, 40, T).astype(np.float32) * np.float32(2.0 ** -24)
    s[1, :] = (s[1] > np.quantile(s[1], 0.95)).astype(np.float32)         # the cut lies among the zeros
    s[2, :] *= 40.0                                                       # far outside the cosine range
    gp = scores_only_problem(T, B, n_kv)
    gp.p.score_mode = {"cosine": api.SCORE_COSINE, "dot": api.SCORE_DOT}[mode]
    gp.scores[0] = torch.from_numpy(s).cuda()
    api.quoka_select_keys(gp.p, gp.scores, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    want = O.select_keys(s.astype(np.float64), B)
    np.testing.assert_array_equal(gp.k_idx[0, :, :B].cpu().numpy(), want)
    assert int(gp.k_cnt[0]) == B


# ---------------------------------------------------------------- full-size configurations
def test_llama8b_32k_full_size():
    w = synth.WORKLOADS["llama8b_32k"]
    gp = problem(0, n_q=w["n_q"], n_kv=w["n_kv"], d=w["d"], T=w["T"], C=w["C"], n_retain=w["n_retain"],
                 kv_budget=w["kv_budget"])
    gp.run_staged()
    stats = check_chain(gp)                 # every stage in full, attention on ALL 32 x 2048 rows
    staged = gp.out.clone()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(staged, gp.out)
    print("llama8b_32k parity stats", stats)


def test_dense_chunk_attention_llama8b_32k_full_size():
    """The dense chunk kernel (Eq. 2), the denominator of every speed-up, at the size the benchmark times it:
    272 key tiles per CTA.  Rows at every tile edge of every head plus random rows, one by one against the oracle."""
    w = synth.WORKLOADS["llama8b_32k"]
    gp = problem(0, n_q=w["n_q"], n_kv=w["n_kv"], d=w["d"], T=w["T"], C=w["C"], n_retain=w["n_retain"],
                 kv_budget=w["kv_budget"])
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    assert api.quoka_last_device_status(gp.ws) == 0
    q, k, v, T = gp.oracle_inputs(0)
    heads, rows = stratified_rows(gp.n_q, gp.C, 256, 77)
    want = O.sparse_attention_rows(q, k, v, T, [np.arange(T)] * gp.n_kv, heads, rows)
    check_attention(f64(gp.out[0])[heads, rows], want, "bf16")


def test_long_128k_full_size():
    w = synth.WORKLOADS["long_128k"]
    gp = problem(0, n_q=w["n_q"], n_kv=w["n_kv"], d=w["d"], T=w["T"], C=w["C"], n_retain=w["n_retain"],
                 kv_budget=w["kv_budget"])
    gp.run_staged()
    stats = check_chain(gp, attn_rows=256)
    print("long_128k parity stats", stats)


def test_serving_mix_paged_full_size():
    w = synth.WORKLOADS["serving_mix"]
    lens = synth.serving_mix_ctx_lens(0, w["batch"])
    gp = problem(0, batch=w["batch"], n_q=w["n_q"], n_kv=w["n_kv"], d=w["d"], T=lens, C=w["C"],
                 n_retain=w["n_retain"], kv_budget=0, budget_frac=w["budget_frac"], paged=True)
    gp.run_staged()
    stats = check_chain(gp, attn_rows=256)
    print("serving_mix parity stats", stats)


SWEEP_BASE = dict(budget_frac=0.12, C=2048, d=128, G=4, n_retain=128)
SWEEP_POINTS = [dict()] + [dict(budget_frac=f) for f in (0.05, 0.25, 0.5)] + [dict(C=c) for c in (512, 8192)] + \
    [dict(d=64)] + [dict(G=g) for g in (1, 8)] + [dict(n_retain=n) for n in (32, 512)] + \
    [dict(budget_frac=0.05, C=512, d=64, G=8, n_retain=32), dict(budget_frac=0.5, C=8192, d=128, G=1, n_retain=512),
     dict(budget_frac=0.5, C=512, d=64, G=1, n_retain=512), dict(budget_frac=0.05, C=8192, d=128, G=8, n_retain=32)]


@pytest.mark.parametrize("pt", SWEEP_POINTS, ids=lambda p: "-".join(f"{k}{v}" for k, v in p.items()) or "base")
def test_sweep_points_32k(pt):
    c = dict(SWEEP_BASE, **pt)
    gp = problem(0, n_q=32, n_kv=32 // c["G"], d=c["d"], T=32768, C=c["C"], n_retain=c["n_retain"], kv_budget=0,
                 budget_frac=c["budget_frac"])
    gp.run_staged()
    check_chain(gp, attn_rows=256)


# ---------------------------------------------------------------- Algorithm 2 as a loop over chunks, eager and as one CUDA graph
def test_chunk_loop_replayed_from_a_cuda_graph_matches_eager_calls():
    # the same buffers serve every chunk; only the cached length (a device tensor) and the host bound change
    T_max, C = 1536, 256
    inp = synth.make_chunk_inputs(12, 1, 8, 2, 128, T_max, C, "bf16")
    gp = GpuProblem(inp, 32, kv_budget=0, budget_frac=0.25)
    lens = [0, 512, 1024, 1536]
    ps = [api.make_params(gp.q, gp.k, gp.out, gp.ctx_len, n_retain=32, budget_frac=0.25, max_ctx_len=t) for t in lens]
    len_dev = [torch.tensor([t], dtype=torch.int32, device="cuda") for t in lens]
    outs = [torch.zeros_like(gp.out) for _ in lens]

    def run():
        for i in range(len(lens)):
            gp.ctx_len.copy_(len_dev[i])
            api.quoka_prefill_chunk(ps[i], gp.q, gp.k, gp.v, gp.out, None, None, gp.ws)
            outs[i].copy_(gp.out)

    run()
    torch.cuda.synchronize()
    want = [o.clone() for o in outs]
    # chunk 0 (empty cache) is plain causal self-attention over rows [0, C): checked against the oracle
    q = f64(gp.inp.q[0])
    dense0, _ = O.dense_chunk_attention(q, f64(gp.inp.k[0, :, :C]), f64(gp.inp.v[0, :, :C]), 0)
    check_attention(f64(want[0][0]), dense0, "bf16")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        run()
        side.synchronize()
        with torch.cuda.graph(g, stream=side):
            run()
    torch.cuda.synchronize()
    for o in outs:
        o.zero_()
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(outs, want):
        assert torch.equal(a, b)
    assert api.quoka_last_device_status(gp.ws) == 0


# ---------------------------------------------------------------- outputs of magnitude 4 and more
def test_large_outputs_are_judged_by_their_bf16_spacing():
    """Two seeded shapes from a randomised soak whose largest deviations are 0.026 on an output of size 4.6 and
    0.020006 on one of size 3.33: above the stated 2e-2, inside half a bf16 spacing of the stored value plus the bf16
    softmax weights' share (tests.parity.attention_bound).  Every element beyond 2e-2 is such a large output."""
    for seed, batch, n_q, n_kv, d, T, C_, n_retain, kv_budget in [(9116, 2, 8, 2, 128, [1100, 63], 700, 4, 128),
                                                                  (9019, 3, 16, 4, 64, [128, 63, 63], 700, 128, 1000)]:
        inp = synth.make_chunk_inputs(seed, batch, n_q, n_kv, d, T, C_, "bf16")
        gp = GpuProblem(inp, n_retain, kv_budget=kv_budget)
        gp.run_staged()
        stats = check_chain(gp)
        assert stats["big_outputs"] > 0, "the shape was chosen because some outputs are large"
        n_over = 0
        for s_ in range(gp.b):
            q, k, v, T_s = gp.oracle_inputs(s_)
            B = O.key_budget(T_s, gp.kv_budget, gp.budget_frac)
            k_idx = gp.k_idx[s_].cpu().numpy()
            want, _ = O.sparse_attention(q, k, v, T_s, [k_idx[kv, :B] for kv in range(gp.n_kv)])
            over = np.abs(f64(gp.out[s_]) - want) > 2e-2
            n_over += int(over.sum())
            assert (np.abs(want[over]) > 3.12).all()
        assert n_over > 0, "the shape was chosen because it exceeds the stated 2e-2 somewhere"
        print("large-output stats", seed, stats, "elements beyond 2e-2:", n_over)


# ---------------------------------------------------------------- query ranking beyond the shared-memory staging limit
def test_f32_chunk_of_8192_queries_ranks_without_staging():
    gp = problem(17, n_q=2, n_kv=1, d=128, T=300, C=8192, dtype="f32", n_retain=100, kv_budget=64)
    gp.run_staged()
    check_chain(gp, attn_rows=64)


# ---------------------------------------------------------------- back-to-back fused calls on one workspace
@pytest.mark.parametrize("C,T", [(200, [150, 90]), (1, [64, 7]), (130, [0, 0])])
def test_back_to_back_fused_calls_when_the_budget_covers_every_cache(C, T):
    """With T_s <= B_s for every sequence the selection kernel has nothing to select; the call must still be
    ordered like a single kernel towards the next call on the same workspace (which rewrites the ranks and
    Q-bar while nothing of this call may still be running)."""
    gp = problem(18, batch=2, n_q=8, n_kv=2, T=T, C=C, n_retain=16, kv_budget=256)
    gp.run_staged()
    want, want_idx = gp.out.clone(), gp.k_idx.clone()
    outs = [torch.zeros_like(gp.out) for _ in range(6)]
    idxs = [torch.full_like(gp.k_idx, -9) for _ in range(6)]
    cnts = [torch.full_like(gp.k_cnt, -9) for _ in range(6)]
    for o, i, c in zip(outs, idxs, cnts):
        api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, o, i, c, gp.ws)
    torch.cuda.synchronize()
    for o, i, c in zip(outs, idxs, cnts):
        assert torch.equal(o, want) and torch.equal(i, want_idx) and torch.equal(c, gp.k_cnt)
    assert api.quoka_last_device_status(gp.ws) == 0


# ------------------------------------------------------------------ split attention (grids far smaller than the GPU)
# With few heads and a short chunk the tensor-core attention kernel cuts every row block's key tiles into parts, one
# CTA each; the parts leave partial results (reference point, sum, un-normalised output) and whichever finishes last
# adds them up in part order.  Shapes below: 8 query heads x 1 row block x batch = 8..16 CTAs before the split, 29-33
# key tiles, so four parts; a short sequence next to a long one gives parts with no tile at all.
@pytest.mark.gpu
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("T,C", [(4100, 200), ([4100, 300], 129), ([3000, 0, 4000], 256)])
def test_split_attention_sparse_against_the_oracle(T, C, paged):
    batch = len(T) if isinstance(T, list) else 1
    gp = problem(31, batch=batch, n_q=8, n_kv=2, T=T, C=C, n_retain=16, kv_budget=0, budget_frac=0.9, paged=paged)
    gp.run_staged()
    check_chain(gp)          # every row of every head, lse included
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)          # same parts, added in the same order
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("T,C", [(4100, 200), ([4100, 300], 129)])
def test_split_attention_dense_against_the_oracle(T, C):
    batch = len(T) if isinstance(T, list) else 1
    gp = problem(32, batch=batch, n_q=8, n_kv=2, T=T, C=C)
    for rep in range(2):     # twice: the arrival counters must be back at zero after a launch
        gp.out.zero_()
        api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
        torch.cuda.synchronize()
        for s in range(batch):
            q, k, v, Ts = gp.oracle_inputs(s)
            want, lse = O.dense_chunk_attention(q, k, v, Ts)
            check_attention(f64(gp.out[s]), want, "bf16")
            assert np.abs(f64(gp.lse[s]) - lse).max() <= 2e-3
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("d,n_q,n_kv", [(64, 8, 2), (64, 4, 4), (64, 6, 2), (128, 4, 4), (128, 6, 2)])
def test_split_attention_in_the_one_cta_kernel(d, n_q, n_kv):
    # head_dim 64 with four, one and three query heads per KV head: parts of one Q tile.  At head_dim 128 these are clusters
    # of pairs; FORMS has the one-CTA kernel's parts
    gp = problem(33, batch=2, n_q=n_q, n_kv=n_kv, d=d, T=[4100, 300], C=200, n_retain=16, kv_budget=0, budget_frac=0.9)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    for s in range(2):
        gp.out.zero_()
        api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
        torch.cuda.synchronize()
        q, k, v, Ts = gp.oracle_inputs(s)
        want, lse = O.dense_chunk_attention(q, k, v, Ts)
        check_attention(f64(gp.out[s]), want, "bf16")
        assert np.abs(f64(gp.lse[s]) - lse).max() <= 2e-3
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
def test_f32_rows_that_one_key_dominates_keep_the_thousands_of_small_weights():
    """A shape from a randomised soak: f32, 5000 listed rows, and chunk rows whose softmax puts 0.99 on one key.
    Summed one by one in fp32, the other 5000 weights (each below half an ulp of the running sum) vanished, 5e-5 of
    the denominator and 2.6e-4 of an output of size 3.1; the scalar kernel's sums are compensated since."""
    inp = synth.make_chunk_inputs(20062, 2, 4, 2, 64, [9000, 63], 200, "f32")
    gp = GpuProblem(inp, 1, 5000, 0.0)
    gp.run_staged()
    check_chain(gp)
    s = 0
    q, k, v, T = gp.oracle_inputs(s)
    cnt = int(gp.k_cnt[s])
    idx = gp.k_idx[s].cpu().numpy()[:, :cnt]
    want, lse = O.sparse_attention(q, k, v, T, [idx[kv] for kv in range(idx.shape[0])])
    assert np.abs(f64(gp.out[s]) - want).max() <= 2e-5       # ten times inside the f32 tolerance
    assert np.abs(f64(gp.lse[s]) - lse).max() <= 1e-5


@pytest.mark.gpu
@pytest.mark.parametrize("n_q,n_kv,d,T,C,frac,paged,fac", [
    (8, 2, 128, 4100, 300, 0.9, False, 6.0),       # CTA pairs, split into parts
    (4, 4, 128, 3000, 257, 0.5, True, 8.0),        # one query head per KV head, paged
    (8, 2, 64, 2500, 200, 0.9, False, 6.0),        # head_dim 64
    (32, 8, 128, 3000, 512, 0.3, False, 5.0)])     # row blocks of one Q tile per CTA, unsplit
def test_logits_far_beyond_the_lazy_rescale_threshold(n_q, n_kv, d, T, C, frac, paged, fac):
    """The tensor-core kernels move the reference point of their exponentials (and rescale the accumulator in
    tensor memory) only when a row's maximum outgrows it by 2^32.  Unit-variance inputs never get there, so here
    the queries are scaled up and the keys grow along the cache: one row's logits span several hundred powers of
    two and the maximum climbs from tile to tile, which also gives the parts of a split launch reference points
    hundreds of powers of two apart."""
    inp = synth.make_chunk_inputs(705, 1, n_q, n_kv, d, T, C, "bf16")
    inp.q = (inp.q.float() * fac).to(torch.bfloat16)
    ramp = torch.linspace(0.5, fac, inp.k.shape[2]).view(1, 1, -1, 1)
    inp.k = (inp.k.float() * ramp).to(torch.bfloat16)
    if paged:
        inp = synth.to_paged(inp, 5)
    gp = GpuProblem(inp, 16, 0, frac, paged=paged)
    q, k, v, Ts = gp.oracle_inputs(0)
    span = (q[0, -1] @ k[0, :Ts + C].T) / np.sqrt(d) * 1.4427
    assert span.max() - span.min() > 300           # powers of two, far beyond the threshold of 32
    gp.run_staged()
    check_chain(gp)
    gp.out.zero_()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    want, lse = O.dense_chunk_attention(q, k, v, Ts)
    check_attention(f64(gp.out[0]), want, "bf16")
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3 * max(1.0, np.abs(lse).max() / 50)
    assert api.quoka_last_device_status(gp.ws) == 0


def _equal_queries(inp): inp.q[:] = inp.q[:, :, :1]
def _equal_keys(inp): inp.k[:, :, :2000] = inp.k[:, :, :1]
def _zero_keys(inp): inp.k[:, :, 100:900] = 0
def _zero_queries(inp): inp.q[:, 0] = 0
def _zero_values(inp): inp.v[:] = 0
def _tiny_keys(inp): inp.k[:, :, :2000] = inp.k[:, :, :2000] * 1e-3


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("mutate", [_equal_queries, _equal_keys, _zero_keys, _zero_queries, _zero_values, _tiny_keys],
                         ids=lambda f: f.__name__.strip("_"))
def test_degenerate_inputs(mutate, dtype):
    """Inputs on which the method's quantities tie or vanish: every query of a head equal (all cosines to the mean
    query tie: ranks by position), every cached key equal (all scores tie: lowest positions first), keys and queries
    of norm zero (the eps of the normalisation decides), values all zero, keys a thousand times smaller than queries."""
    inp = synth.make_chunk_inputs(800, 1, 8, 2, 128, 2000, 300, dtype)
    mutate(inp)
    gp = GpuProblem(inp, 16, 300, 0.0)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    assert torch.isfinite(gp.out.float()).all()
    assert api.quoka_last_device_status(gp.ws) == 0


def _token_major(t):            # (b, heads, rows, d) view of a (b, rows, heads, d) buffer
    return t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)


def _padded_rows(t, pad):       # rows `pad` elements longer than head_dim
    big = torch.zeros(*t.shape[:3], t.shape[3] + pad, dtype=t.dtype, device=t.device)
    big[..., : t.shape[3]] = t
    return big[..., : t.shape[3]]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("layout", ["token-major", "padded"])
@pytest.mark.parametrize("n_q,n_kv,d,T,C,frac", [(8, 2, 128, [4100, 700], 129, 0.9), (4, 4, 64, 1500, 200, 0.3),
                                                 (32, 8, 128, 2000, 512, 0.12)])
def test_strided_layouts(n_q, n_kv, d, T, C, frac, layout, dtype):
    """q, out and the KV cache are described by element strides: the same problem with queries and cache stored
    token-major ((b, rows, heads, d), the layout projections usually write) and with padded rows."""
    batch = len(T) if isinstance(T, list) else 1
    inp = synth.make_chunk_inputs(900, batch, n_q, n_kv, d, T, C, dtype)
    gp = GpuProblem(inp, 16, 0, frac)
    fq, fk = (_token_major, _token_major) if layout == "token-major" else (lambda t: _padded_rows(t, 64), lambda t: _padded_rows(t, 8))
    gp.q, gp.out = fq(gp.q), fq(torch.zeros_like(gp.q))
    gp.k, gp.v = fk(gp.k), fk(gp.v)
    assert not gp.q.is_contiguous() and not gp.k.is_contiguous()
    gp.p = api.make_params(gp.q, gp.k, gp.out, gp.ctx_len, n_retain=16, kv_budget=0, budget_frac=frac, max_ctx_len=gp.max_ctx)
    gp.run_staged()
    check_chain(gp)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n_q,n_kv,d,T,C", [(8, 2, 128, 3000, 300), (4, 4, 64, 1500, 200), (8, 2, 128, 4100, 1)])
@pytest.mark.parametrize("scale", [0.03, 0.3])
def test_softmax_scale_given_by_the_caller(scale, n_q, n_kv, d, T, C, dtype):
    """softmax_scale != 0 replaces 1 / sqrt(head_dim) in Eq. 1 / Eq. 2 (every attention kernel: CTA pairs, one CTA,
    scalar, and the one-query kernel), and does not touch the selection."""
    inp = synth.make_chunk_inputs(950, 1, n_q, n_kv, d, T, C, dtype)
    gp = GpuProblem(inp, 16, 0, 0.5)
    gp.p.softmax_scale = scale
    gp.run_staged()
    q, k, v, Ts = gp.oracle_inputs(0)
    cnt = int(gp.k_cnt[0])
    idx = gp.k_idx[0].cpu().numpy()[:, :cnt]
    want, lse = O.sparse_attention(q, k, v, Ts, [idx[kv] for kv in range(n_kv)], scale=scale)
    check_attention(f64(gp.out[0]), want, dtype)
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3
    sel_scaled = gp.k_idx.clone()
    gp.p.softmax_scale = 0.0
    gp.run_staged()
    assert torch.equal(gp.k_idx, sel_scaled)
    gp.p.softmax_scale = scale
    gp.out.zero_()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    want, lse = O.dense_chunk_attention(q, k, v, Ts, scale=scale)
    check_attention(f64(gp.out[0]), want, dtype)
    assert np.abs(f64(gp.lse[0]) - lse).max() <= 2e-3


@pytest.mark.gpu
def test_split_attention_over_a_200k_row_cache():
    # 8 heads x 1 row block = 8 CTAs before the split, 782 list tiles: eight parts of ~100 tiles each
    inp = synth.make_chunk_inputs(970, 1, 8, 2, 128, 200000, 256, "bf16")
    gp = GpuProblem(inp, 32, 0, 0.5)
    gp.run_staged()
    check_chain(gp, attn_rows=48)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    assert api.quoka_last_device_status(gp.ws) == 0


@pytest.mark.gpu
def test_split_attention_of_a_grid_between_half_a_wave_and_a_wave():
    # 8 heads x 10 row blocks = 80 CTAs of ~130 tiles: three parts each (two waves of a third beat one wave of a whole)
    inp = synth.make_chunk_inputs(971, 1, 8, 2, 128, 17000, 2560, "bf16")
    gp = GpuProblem(inp, 64, 0, 0.9)
    gp.run_staged()
    check_chain(gp, attn_rows=64)
    staged = gp.out.clone()
    gp.out.zero_()
    api.quoka_prefill_chunk(gp.p, gp.q, gp.k, gp.v, gp.out, gp.k_idx, gp.k_cnt, gp.ws)
    torch.cuda.synchronize()
    assert torch.equal(gp.out, staged)
    gp.out.zero_()
    api.quoka_dense_chunk_attn(gp.p, gp.q, gp.k, gp.v, gp.out, gp.lse, gp.ws)
    torch.cuda.synchronize()
    q, k, v, Ts = gp.oracle_inputs(0)
    heads, rows = stratified_rows(8, 2560, 48, 3)
    idx_all = [np.arange(Ts)] * 2
    want = O.sparse_attention_rows(q, k, v, Ts, idx_all, heads, rows)       # every cached row listed = Eq. 2
    check_attention(f64(gp.out[0])[heads, rows], want, "bf16")
    assert api.quoka_last_device_status(gp.ws) == 0
