"""GPU parity for the selection scopes other than one list per KV head (paper Sec. 3.1: importance is
predicted per head; App. "additional evaluation": a head-less predictor, one importance per token and
layer): one list per query head, one list per layer.  The oracle needs no new arithmetic for them: a
per-query-head unit is a group of one whose keys are its KV head's, and a per-layer unit scores the
[Hkv*D] x d' projection of the concatenated key and hands its one list to every head."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2503_07518_b200 import workloads as wl  # noqa: E402
from test_gpu_parity import H, full_pipeline_check, tb  # noqa: E402,F401


CASES = [
    # a block per list, or a small cluster; bf16 tensor-core attention with a group of one / of four
    (2, dict(n_layers=2, batch=2, lengths=[5000, 777], budget=200, sinks=3, recent=9)),
    # fp32 storage, d' = 16, g = 2
    (1, dict(n_layers=1, n_q_heads=8, n_kv_heads=4, imp_dim=16, batch=3, lengths=[1500, 260, 2049], budget=100, sinks=1, recent=4)),
]


@pytest.mark.parametrize("scope", [1, 2])
@pytest.mark.parametrize("ci", range(len(CASES)))
def test_scope_pipeline_matches_oracle(H, scope, ci):
    """Projection (per-layer scope: summed over the KV heads), selection and attention from the stored
    lists, dense attention too, with and without neighbours and across an append + reuse step."""
    b_ = tb()
    cfg, over = CASES[ci]
    w = wl.workload(cfg, **over)
    case = H.Case(w, max_radius=2, extra_len=4, list_scope=scope)          # Case checks the projection
    assert case.Hl == (w.n_q_heads if scope == 1 else 1) and case.Hi == (w.n_kv_heads if scope == 1 else 1)
    p = b_.select_params(w.budget, w.sinks, w.recent)
    full_pipeline_check(H, case, p, dense_too=True)
    pn = b_.select_params(w.budget, w.sinks, w.recent, radius=2, nmode=b_.TB_NEIGHBOR_DILATE)
    full_pipeline_check(H, case, b_.select_params(w.budget, w.sinks, w.recent, radius=1, nmode=b_.TB_NEIGHBOR_CLUSTER), step=3)
    full_pipeline_check(H, case, pn, step=1)                               # leaves the DILATE lists stored for the reuse step below
    # a decode step that appends and reuses the stored lists (interval 4, step 1)
    case.append_step(0)
    case.project_range(list(case.proj), list(case.cur))
    q, qi = H.queries(w, 2)
    stored = H.gpu_select(case, qi[:, :, :case.Hl * case.gl], b_.select_params(w.budget, w.sinks, w.recent, radius=2, interval=4, step=1))
    out, _ = H.gpu_attention(case, q, pn)
    for l in range(w.n_layers):
        for b in range(w.batch):
            for h in range(case.Ha):
                ref, _ = case.oracle_attention(l, b, h, q[l, b], stored[l][b][h * case.Hl // case.Ha], pn)
                assert np.abs(out[l, b, h * case.ga:(h + 1) * case.ga] - ref).max() <= H.ATTN_TOL[w.dtype]


def test_per_query_head_lists_many_problems(H):
    """One list per query head turns 24 sequences x 32 query heads into 768 problems of one launch:
    a block of 256 threads per list, then attention with a group of one."""
    b_ = tb()
    w = wl.workload(2, n_layers=1, batch=24, lengths=[1800 + 53 * i for i in range(24)], budget=96)
    case = H.Case(w, list_scope=b_.TB_SCOPE_Q_HEAD)
    full_pipeline_check(H, case, b_.select_params(w.budget, w.sinks, w.recent))


def test_per_query_head_lists_reduce_to_group_lists(H):
    """If the g importance queries of every group are equal, a group's sum is g times each of them, so
    per-query-head lists must equal the per-KV-head list of the same inputs (and so must the outputs)."""
    b_ = tb()
    w = wl.workload(2, n_layers=1, batch=2, lengths=[3000, 901], budget=150, sinks=2, recent=6)
    q, qi = H.queries(w)
    qi = np.repeat(qi[:, :, ::w.group], w.group, axis=2)                   # every head of a group gets the group's first query
    p = b_.select_params(w.budget, w.sinks, w.recent)
    kv_case = H.Case(w)
    kv_lists = H.gpu_select(kv_case, qi, p)
    kv_out, _ = H.gpu_attention(kv_case, q, p)
    q_case = H.Case(w, list_scope=b_.TB_SCOPE_Q_HEAD)
    q_lists = H.gpu_select(q_case, qi, b_.select_params(w.budget, w.sinks, w.recent, reduce=b_.TB_PER_QHEAD))
    q_out, _ = H.gpu_attention(q_case, q, p)
    for b in range(w.batch):
        for hq in range(w.n_q_heads):
            assert np.array_equal(q_lists[0][b][hq], kv_lists[0][b][hq // w.group])
    assert np.abs(q_out - kv_out).max() <= H.ATTN_TOL[w.dtype]


def test_scope_argument_checks(H):
    b_ = tb()
    w = wl.workload(2, n_layers=1, batch=1, lengths=[600], budget=32)
    case = H.Case(w)                                                      # lists per KV head
    _, qi = H.queries(w)
    with pytest.raises(b_.TBError) as e:
        H.gpu_select(case, qi, b_.select_params(w.budget, w.sinks, w.recent, reduce=b_.TB_PER_QHEAD))
    assert e.value.status == b_.TB_ERR_UNSUPPORTED
    cfg = b_.tb_config(1, 8, 8, 128, 32, b_.TB_BF16, 1, 256, 16, 0, 0, 7)  # no such scope
    sizes = [ctypes.c_size_t() for _ in range(4)]
    assert b_.lib().tb_query_sizes(ctypes.byref(cfg), *[ctypes.byref(x) for x in sizes]) == b_.TB_ERR_INVALID_ARG
    # sizes follow the scope: per-layer keeps one projected key per token, per-query-head g times the lists
    def sizes_of(scope):
        c = b_.tb_config(2, 32, 8, 128, 32, b_.TB_BF16, 2, 4096, 256, 0, 0, scope)
        out = [ctypes.c_size_t() for _ in range(4)]
        assert b_.lib().tb_query_sizes(ctypes.byref(c), *[ctypes.byref(x) for x in out]) == b_.TB_OK
        return [x.value for x in out]
    kvh, qh, lay = sizes_of(0), sizes_of(1), sizes_of(2)
    assert kvh[0] == qh[0] == lay[0] and kvh[1] == qh[1] == 8 * lay[1]
    assert qh[2] > kvh[2] > lay[2]


@pytest.mark.parametrize("q_heads,kv_heads,dp", [(4, 2, 32), (8, 2, 16), (7, 1, 32), (8, 1, 32), (3, 1, 16)])
def test_lists_that_share_a_key_stream(H, q_heads, kv_heads, dp):
    """Few per-query-head lists: lengths off a 32-row group, a sequence short enough to be unsampled beside a long one, both
    neighbour rules, and thresholds in crowded bins (massive ties).  Each list streams its keys itself at this number; the kernel
    that reads a stream once for all its lists is in test_gpu_select_routes.py."""
    for lengths, budget, sinks, recent, radius, nmode in (([9001, 700], 300, 2, 5, 0, 0), ([12345, 8300], 1000, 0, 0, 1, 1), ([40007], 5, 0, 16, 2, 0)):
        w = wl.workload(2, n_layers=1, n_q_heads=q_heads, n_kv_heads=kv_heads, imp_dim=dp, batch=len(lengths), lengths=lengths, budget=budget,
                        sinks=sinks, recent=recent, radius=radius, nmode=nmode)
        case = H.Case(w, list_scope=tb().TB_SCOPE_Q_HEAD)
        p = tb().select_params(budget, sinks, recent, radius, nmode)
        full_pipeline_check(H, case, p)
        _, qi = H.queries(w)
        for ties in (np.zeros_like(qi), np.where(np.arange(dp) == 0, np.float32(1), np.float32(0)) * np.ones_like(qi)):
            if ties.any():                             # few distinct scores: the first channel of every key is 0, 1 or 2
                for b, L in enumerate(lengths):
                    v = (np.arange(L) * 7919 % 3).astype(np.float32)
                    case.Kimp[0][b][:, :L, 0] = wl.to_storage(v, w.dtype)
                    case.ctx.kimp[0, b, :, :L] = H.to_dev(case.Kimp[0][b][:, :L], w.dtype)
            lists = H.gpu_select(case, ties, p)
            assert case.ctx.get_status() == 0
            for b in range(w.batch):
                for h in range(q_heads):
                    _, full, _ = case.oracle_select(0, b, h, ties[0, b], p)
                    assert np.array_equal(lists[0][b][h], full)


@pytest.mark.parametrize("dp", [16, 32])
@pytest.mark.parametrize("scope,reduce,lengths", [(0, 0, [700, 40]), (0, 1, [700, 300]), (0, 0, [3000]), (1, 0, [700]), (1, 0, [12001, 700])])
def test_infinite_scores_rank_as_infinities(H, scope, reduce, lengths, dp):
    """A projected key or a query that overflowed to an infinity gives infinite scores: last or first in the ranking, equal
    ones by position, whichever kernel ranks them.  (No term of a score is inf * 0 here, no sum inf - inf.)"""
    w = wl.workload(2, n_layers=1, n_q_heads=8, n_kv_heads=2, imp_dim=dp, batch=len(lengths), lengths=lengths, budget=max(lengths) - 30)
    case = H.Case(w, list_scope=scope)
    _, qi = H.queries(w)
    qi = np.abs(qi) + np.float32(0.01)                 # the key's sign is the infinity's; three bf16 terms, some of them negative
    r = np.random.Generator(np.random.PCG64(3))
    for b, L in enumerate(lengths):
        x = wl.storage_to_f32(case.Kimp[0][b][:, :L], w.dtype).copy()
        x[x == 0] = 1.0
        for h in range(2):
            rows = r.permutation(L)[:L // 5 + 2]
            x[h, rows, r.integers(0, dp, rows.size)] = np.where(np.arange(rows.size) % 7 == 0, np.inf, -np.inf)
        case.Kimp[0][b][:, :L] = wl.to_storage(x.astype(np.float32), w.dtype)
        case.ctx.kimp[0, b, :, :L] = H.to_dev(case.Kimp[0][b][:, :L], w.dtype)
    heads = np.arange(8) % 4 == 2                      # one head of a group asks for an infinity in a channel of its own
    for queries in (qi, np.where(heads[None, None, :, None] & (np.arange(dp) == 3), np.float32(np.inf), qi)):
        if not np.isfinite(queries).all():             # ... of keys that are finite and not zero
            for b, L in enumerate(lengths):
                x = r.standard_normal((2, L, dp)).astype(np.float32)
                x[np.abs(x) < 0.01] = 1.0
                case.Kimp[0][b][:, :L] = wl.to_storage(x, w.dtype)
                case.ctx.kimp[0, b, :, :L] = H.to_dev(case.Kimp[0][b][:, :L], w.dtype)
        for budget in (5, min(lengths) // 2, w.budget):
            p = tb().select_params(budget, reduce=reduce)
            lists = H.gpu_select(case, queries, p)
            assert case.ctx.get_status() == 0
            for b in range(w.batch):
                for h in range(case.Hl):
                    _, full, s = case.oracle_select(0, b, h, queries[0, b], p)
                    assert not np.isnan(s).any()
                    H.check_selection(lists[0][b][h], full, s)


@pytest.mark.parametrize("n_heads,batch,length", [(4, 1, 12000), (8, 2, 10300), (8, 20, 9000), (8, 10, 12000), (2, 1, 3000)])
def test_asking_for_the_lists_does_not_change_them(H, n_heads, batch, length):
    """Keys that are permutations of one another under a query of equal entries: exact scores tie, fp32 sums differ in their
    last bits by the order of summation.  The stored list has to be the same whether a copy is asked for or not."""
    dp = 32
    ctx = tb().Context(1, n_heads, n_heads, 128, dp, tb().TB_BF16, batch, length, 500)
    zeros = torch.zeros(batch * length, n_heads, 128, dtype=torch.bfloat16, device="cuda")
    ctx.append_kv(0, 1, None, [length] * batch, zeros, zeros)
    ctx.project_keys(0, 1, None, [0] * batch, [length] * batch)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    row = torch.randn(dp, generator=gen, device="cuda").to(torch.bfloat16)
    perm = torch.rand(ctx.kimp.shape, generator=gen, device="cuda").argsort(-1)
    ctx.kimp.copy_(row[perm])
    q = torch.full((1, batch, n_heads, dp), 1.0 / 3.0, device="cuda")
    idx = torch.zeros(2, 1, batch, n_heads, ctx.index_capacity, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(2, 1, batch, n_heads, dtype=torch.int32, device="cuda")
    refresh, stored = tb().select_params(500, interval=2), tb().select_params(500, interval=2, step=1)
    ctx.select_topk(0, 1, None, batch, q, refresh)
    ctx.select_topk(0, 1, None, batch, q, stored, idx[0], cnt[0])
    ctx.select_topk(0, 1, None, batch, q, refresh, idx[1], cnt[1])
    assert ctx.get_status() == 0 and (cnt == 500).all()
    assert torch.equal(idx[0], idx[1])
    assert not torch.equal(idx[0][..., :500], torch.arange(500, device="cuda", dtype=torch.int32).expand(1, batch, n_heads, 500))
