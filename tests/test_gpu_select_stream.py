"""The selection kernels that load rows straight into registers, at the sizes where they can go wrong: shares of a cluster, rows
past the last whole group of 32, ragged batches with problems that have nothing to rank, blocks that keep digits instead of
scores, the block sizes, crowded bins, ties and infinities; one list per KV head, and one per query head.  Keys and queries are small whole numbers, so every score is exact and every list is the
oracle's, whatever the order of the sums."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from test_gpu_parity import H, tb  # noqa: E402,F401

# heads, group, lengths, d', dtype, reduce, budget, sinks, recent, radius, mode, data
CASES = [
    (1, 1, [10241], 32, "bf16", "sum", 700, 0, 0, 0, 0, "int"),                    # ten blocks, one row past a group
    (2, 4, [12345, 10500, 3, 700], 32, "bf16", "sum", 900, 4, 16, 0, 0, "int"),    # ragged: everything, and less than a block's share
    (8, 4, [32768], 32, "bf16", "max", 3276, 0, 0, 0, 0, "int"),
    (8, 1, [16411, 16384], 16, "bf16", "sum", 300, 16, 64, 1, 0, "int"),           # neighbours across the blocks' borders
    (4, 2, [20000, 11111], 32, "fp32", "sum", 2000, 3, 5, 2, 1, "int"),
    (4, 8, [15001], 16, "fp32", "max", 7000, 0, 0, 0, 0, "int"),                   # threshold near zero score
    (8, 4, [11000] * 20, 32, "bf16", "sum", 1100, 0, 0, 1, 1, "int"),              # 160 problems: blocks of 256 threads
    (8, 1, [21003] + [17000] * 19, 32, "bf16", "sum", 3000, 0, 0, 0, 0, "int"),    # ... that keep digits
    (8, 1, [2050] * 20, 32, "fp32", "sum", 200, 0, 0, 0, 0, "int"),
    (8, 1, [47009] * 10, 32, "bf16", "sum", 5000, 0, 0, 0, 0, "int"),              # one block of 512 threads, digits
    (8, 1, [50000, 49999] * 14, 16, "bf16", "sum", 5000, 0, 0, 1, 0, "int"),       # two waves of those
    (2, 4, [40000], 32, "bf16", "sum", 1234, 0, 0, 0, 0, "ties"),
    (8, 1, [47000] * 10, 16, "bf16", "max", 2345, 0, 0, 0, 0, "ties"),             # ... from the rows again
    (2, 1, [30000], 32, "fp32", "sum", 29990, 0, 0, 0, 0, "ties"),
    (2, 2, [30000], 32, "bf16", "sum", 40, 0, 0, 0, 0, "outliers"),                # the sampled bracket ends far below the threshold
    (8, 1, [47000] * 10, 32, "bf16", "sum", 100, 0, 0, 0, 0, "outliers"),
    (2, 2, [20000], 32, "bf16", "sum", 50, 0, 0, 0, 0, "inf"),
    (2, 2, [20000], 16, "bf16", "max", 50, 0, 0, 0, 0, "inf"),
    # short lists, blocks of 256 threads: two per SM and more (and, with one of 5003, the kernel that parks its keys)
    (8, 2, [2048, 33, 1000, 64] * 5, 32, "bf16", "sum", 100, 2, 3, 1, 0, "int"),
    (8, 1, [5003, 4000, 1, 31, 257] * 8, 32, "bf16", "sum", 400, 0, 0, 0, 0, "int"),
    (8, 4, [1300] * 38, 16, "bf16", "max", 600, 0, 16, 2, 1, "int"),
    (8, 1, [3000] * 38, 32, "bf16", "sum", 700, 0, 0, 0, 0, "ties"),
    (8, 1, [3000] * 38, 32, "bf16", "sum", 90, 0, 0, 0, 0, "outliers"),
    (8, 2, [2500] * 38, 32, "bf16", "sum", 50, 0, 0, 0, 0, "inf"),
    # one list per query head
    (4, 7, [8200] * 11, 32, "bf16", "per head", 500, 4, 0, 1, 1, "int"),
    (8, 4, [15000], 32, "bf16", "per head", 900, 0, 0, 0, 0, "int"),
    (4, 4, [11000, 10500] * 5, 16, "bf16", "per head", 800, 0, 0, 0, 0, "int"),
    # infinities of either sign, an infinite query, NaN: where scores are kept, and where digits are
    (2, 2, [20000], 32, "bf16", "sum", 900, 0, 0, 0, 0, "infs"),
    (2, 2, [20000], 16, "bf16", "max", 19900, 0, 0, 0, 0, "infs"),
    (2, 4, [20000], 32, "bf16", "max", 9000, 0, 0, 0, 0, "infinite query"),
    (2, 4, [20000], 32, "fp32", "max", 15000, 0, 0, 0, 0, "infinite query"),
    (2, 2, [20000], 32, "fp32", "sum", 19900, 0, 0, 0, 0, "infs"),
    (2, 2, [20000], 32, "bf16", "sum", 900, 0, 0, 0, 0, "nan"),
    (8, 1, [47000] * 10, 32, "bf16", "sum", 700, 0, 0, 0, 0, "infs"),
    (8, 1, [47000] * 10, 16, "bf16", "sum", 46800, 0, 0, 0, 0, "infs"),
    (8, 1, [47000] * 10, 16, "bf16", "max", 5000, 0, 0, 0, 0, "infs"),
    (8, 2, [47000] * 10, 32, "bf16", "max", 12000, 0, 0, 0, 0, "infinite query"),
    (8, 1, [47000] * 10, 32, "bf16", "sum", 700, 0, 0, 0, 0, "nan"),
    (8, 1, [23000] * 10, 32, "fp32", "sum", 700, 0, 0, 0, 0, "infs"),
    (8, 1, [47000] * 10, 32, "bf16", "sum", 30000, 0, 0, 0, 0, "below"),
    (2, 1, [30000], 32, "bf16", "sum", 9000, 0, 0, 0, 0, "binades"),
    # more equal rows at the threshold than are ranked, where digits are kept: one block, two waves of them, a cluster
    (8, 1, [47000, 46001] * 5, 32, "bf16", "sum", 5000, 0, 0, 0, 0, "equal"),
    (8, 1, [50000, 49999] * 14, 16, "bf16", "sum", 5000, 0, 0, 1, 0, "equal"),
    (1, 2, [900001], 32, "bf16", "sum", 50000, 0, 0, 0, 0, "equal"),
    (8, 1, [47000] * 10, 16, "fp32", "sum", 4000, 0, 0, 0, 0, "equal"),
]


@pytest.mark.parametrize("ci", range(len(CASES)))
def test_lists_are_the_oracles(H, ci):
    check_lists(H, CASES[ci], ci)


# one per kernel that selects; their queries are read in different ways
@pytest.mark.parametrize("case", [
    (2, 4, [700, 333], 32, "bf16", "sum", 90, 0, 0, 0, 0, "int"),
    (2, 4, [700, 333], 16, "fp32", "sum", 90, 0, 0, 0, 0, "int"),
    (2, 4, [12345, 10500], 32, "bf16", "sum", 900, 4, 16, 0, 0, "int"),
    (2, 4, [12345, 10500], 16, "bf16", "sum", 900, 4, 16, 1, 0, "int"),
    (2, 4, [12345, 10500], 32, "bf16", "max", 900, 4, 16, 0, 0, "int"),
    (2, 4, [12345, 10500], 32, "fp32", "sum", 900, 4, 16, 0, 0, "int"),
    (2, 8, [12345, 10500], 16, "fp32", "max", 900, 4, 16, 0, 0, "int"),
    (8, 4, [11000] * 20, 32, "bf16", "sum", 1100, 0, 0, 0, 0, "int"),
    (8, 4, [2050] * 20, 32, "fp32", "sum", 200, 0, 0, 0, 0, "int"),
    (8, 1, [9000] * 48, 32, "bf16", "sum", 400, 0, 0, 0, 0, "int"),
    (4, 4, [15000] * 10, 32, "bf16", "per head", 800, 0, 0, 0, 0, "int"),
])
def test_queries_may_start_at_any_float(H, case):
    """The importance queries are floats: a view that starts one float into its storage gives the same lists."""
    check_lists(H, case, 5, q_offset=1)


def check_lists(H, case, seed, q_offset=0, kernel=None, dev_lengths=False):
    """The lists of one call, and of the stored lists after it, are the oracle's; `kernel`: the one that has to select."""
    b_ = tb()
    heads, g, lens, dp, dt, reduce, budget, sinks, recent, radius, mode, data = case
    dtype = b_.TB_BF16 if dt == "bf16" else b_.TB_F32
    store = b_.torch_dtype(dtype)
    red = b_.TB_GROUP_MAX if reduce == "max" else b_.TB_GROUP_SUM
    per_head = reduce == "per head"
    lists, gl = (heads * g, 1) if per_head else (heads, g)
    B = len(lens)
    ctx = b_.Context(1, heads * g, heads, 128, dp, dtype, B, -(-max(lens) // 64) * 64, budget, radius,
                     list_scope=b_.TB_SCOPE_Q_HEAD if per_head else b_.TB_SCOPE_KV_HEAD)
    ctx.set_projection(0, torch.zeros(heads, 128, dp, dtype=store, device="cuda"))
    rows = torch.zeros(sum(lens), heads, 128, dtype=store, device="cuda")
    ctx.append_kv(0, 1, None, lens, rows, rows)
    ctx.project_keys(0, 1, None, [0] * B, lens)
    del rows
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.randn(ctx.kimp.shape, generator=gen, device="cuda")
    x = (x.mul_(1.0).round_() if data == "ties" else x.mul_(40).round_()).clamp_(-120, 120)
    q = torch.randn(1, B, heads * g, dp, generator=gen, device="cuda").mul_(20).round_().clamp_(-60, 60)
    if data == "ties":                                   # whole numbers below 2 dp: thousands share a score
        q = q.sign()
    if data == "outliers":                               # more rows than are wanted score far above all others, close together
        for b, L in enumerate(lens):
            at = torch.randint(0, L, (budget + min(800, L // 4),), generator=gen, device="cuda")
            up = q[0, b].view(heads, g, dp).sum(1).sign().unsqueeze(1) * 120
            x[0, b][:, at] = up + torch.randint(-3, 4, (heads, len(at), dp), generator=gen, device="cuda")
    lo = min(sinks, min(lens))
    if data in ("binades", "below"):                     # one channel carries the score, one head of a group asks for it
        x[..., 1:], x[..., 0] = 0, x[..., 0].bfloat16().float()
        q.view(1, B, lists, gl, dp).copy_((torch.arange(gl * dp, device="cuda") == 0).view(gl, dp))
    if data == "binades":                                # 400 of them, both signs
        x[..., 0] = torch.exp2(torch.randint(-100, 101, x.shape[:-1], generator=gen, device="cuda").float()) * x[..., 0].sign().add(0.5).sign()
    if data == "below":                                  # the rows that are looked at first score highest, the wanted ones do not
        for b, L in enumerate(lens):
            at = lo + torch.arange(64, device="cuda") * max(L - sinks - recent, 1) // 64
            x[0, b, :, at, 0] = 1000 + 8 * torch.arange(64, device="cuda", dtype=torch.float32)
    if data == "infs":                                   # of either sign
        for b, L in enumerate(lens):
            x[0, b, :, 50:L:97, 3] = float("inf")
            x[0, b, :, 90:L:97, 3] = float("-inf")
        q[..., 3] = q[..., 3].abs() + 1
    if data == "infinite query":                         # one head's, of keys that are not zero
        x[..., 3] = torch.where(x[..., 3] == 0, 7, x[..., 3])
        q[:, :, ::gl, 3] = float("inf")
    if data == "equal":                                  # some hundred equal rows at the threshold, in one block's share and all over
        for b, L in enumerate(lens):
            at = torch.cat([torch.arange(L - 400, L, device="cuda"), torch.randint(0, L, (300,), generator=gen, device="cuda")])
            for h in range(heads):
                kth = (x[0, b, h, :L] @ q[0, b, h * g:(h + 1) * g].sum(0)).topk(budget).indices[-1]
                x[0, b, h, at] = x[0, b, h, kth].clone()
    if data == "nan":                                    # takes no number's place
        for b, L in enumerate(lens):
            x[0, b, :, 50:L:97, 3] = float("nan")
    if data == "inf":
        x[0, 0, :, 1000:lens[0]:97, 3] = float("inf")    # of either sign once multiplied: every row's other products are finite
        q[..., 3] = q[..., 3].abs() + 1
    ctx.kimp.copy_(x.to(store))
    q_mem = torch.empty(q.numel() + q_offset, device="cuda")
    q_at = q_mem[q_offset:].view(q.shape).copy_(q)
    idx = torch.zeros(1, B, lists, ctx.index_capacity, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, B, lists, dtype=torch.int32, device="cuda")
    if dev_lengths:
        ctx.use_device_lengths(True)
    if kernel:
        p = b_.select_params(budget, sinks, recent, radius, mode, reduce=red)
        assert kernel in H.launched_kernels(lambda: ctx.select_topk(0, 1, None, B, q_at, p, idx, cnt))[0]
    for copied in (True, False):                         # the caller's copy, and the stored lists
        p = b_.select_params(budget, sinks, recent, radius, mode, 2, 0 if copied else 1, red)
        if copied:
            ctx.select_topk(0, 1, None, B, q_at, p, idx, cnt)
        else:
            idx.zero_(), cnt.zero_()
            ctx.select_topk(0, 1, None, B, None, p, idx, cnt)
        assert ctx.get_status() == 0
        got_n, got = cnt.cpu().numpy(), idx.cpu().numpy()
        for b in range(0, B, 1 if copied else max(1, B - 1)):
            for h in range(lists):
                s = (ctx.kimp[0, b, h * heads // lists, :lens[b]].double() @ q[0, b, h * gl:(h + 1) * gl].double().T)
                s = (s.max(1).values if reduce == "max" else s.sum(1)).cpu().numpy()
                s = np.where(np.isnan(s), -np.inf, s)
                want = H.orc.select(s, sinks, recent, budget)
                lo, hi = H.orc.candidate_range(lens[b], sinks, recent)
                if radius and len(want) < hi - lo:
                    want = H.orc.neighbors(want, radius, mode, lo, hi)
                assert np.array_equal(got[0, b, h, :got_n[0, b, h]], want), (b, h)
