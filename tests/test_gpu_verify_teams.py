"""Verification of batches whose sequences run on teams of CTAs, parts of a team and single CTAs (score-cache kernel):
lengths around the edges of key tiles and of a part's capacity, more rounds than the work table holds, more sequences
than the schedule sorts, many short sequences back to back.  Against the oracle at 2e-3, the bar of every
verification test, and bit for bit between repeated passes (the reductions run in a fixed order)."""
import dataclasses

import pytest
import torch

import oracle
from paper_2607_27735_b200 import binding, inputs
from verify_schedule import TABLE, schedule

pytestmark = pytest.mark.gpu
TOL = 2e-3

SHAPES = [  # (contexts, query heads, KV heads, head_dim, rows, page)
    ([127, 128, 129, 255, 257, 1023, 1025], 8, 2, 128, 5, 0),
    ([9, 4096, 9, 700, 2600], 32, 8, 128, 9, 16),               # one long sequence among short ones; T = n_q
    ([1364, 1200, 1309, 332, 541, 404, 959, 601, 419, 663, 1292, 728], 8, 8, 128, 6, 0),  # a CTA per problem
    ([1792, 1793, 3584, 3585, 7000, 512], 8, 2, 64, 7, 64),      # a part's capacity at 14 tiles, +- 1
    ([300 + 17 * i for i in range(70)], 4, 2, 128, 3, 0),        # more sequences than are sorted
]


def make(ctx, hq, hkv, d, n_q, page, layers=1, seed=1):
    cfg = inputs.small_config(ctx=(min(ctx), max(ctx)), n_q=n_q, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, planted=4,
                              batch=len(ctx), n_layers=layers, page_size=page, shuffled_pages=page > 0, seed=seed)
    return inputs.make_case(cfg, device="cuda", ctx_override=list(ctx))


def check(case, T, out_bf16=False):
    out, lse, stats, ws = binding.spec_verify_attn(case.kv, case.q_verify, case.ctx_len, T, out_bf16=out_bf16)
    assert binding.read_status(ws) == 0
    assert binding.last_verify_impl() == binding.VERIFY_TCGEN05_CACHED
    o_out, o_lse, o_stats = oracle.verify_attn(case.kv.cpu(), case.q_verify.cpu(), case.ctx_len.cpu(), 16, stats.shape[-1])
    # bf16 output: half a step of 2^-8 of the largest value on top
    bar = TOL + (o_out.abs().max().item() * 2.0 ** -8 if out_bf16 else 0.0)
    assert (out.cpu().double() - o_out).abs().max().item() <= bar
    assert (lse.cpu().double() - o_lse).abs().max().item() <= TOL
    for b, t in enumerate(case.ctx_len.tolist()):
        assert (stats[:, b, :, :t].cpu().double() - o_stats[:, b, :, :t]).abs().max().item() <= TOL
    return out, lse, stats, ws


@pytest.mark.parametrize("ctx,hq,hkv,d,n_q,page", SHAPES)
@pytest.mark.parametrize("out_bf16", [False, True])
def test_ragged_batches(ctx, hq, hkv, d, n_q, page, out_bf16):
    check(make(ctx, hq, hkv, d, n_q, page), max(ctx), out_bf16)


@pytest.mark.parametrize("slack", [0, 3000, 60000])
def test_capacity_far_above_the_lengths(slack):
    """The split is sized for the longest context the call allows; the lengths in device memory may be far below."""
    ctx = [700, 3000, 150]
    cap = max(ctx) + slack
    case = make([cap] * 3, 32, 8, 128, 5, 0)
    case = dataclasses.replace(case, ctx_len=torch.tensor(ctx, dtype=torch.int32, device="cuda"))
    check(case, cap)


def test_several_rounds_per_team():
    check(make([4100, 3000, 5000, 4500], 32, 8, 128, 9, 0, layers=6), 5000)


# More units than the work table holds.  "stale": a CTA has nothing to exchange for a stretch of units in which it would
# find, 32 units back, an entry of a problem that it shared (whole teams before parts that leave the last CTA of a team idle;
# with more than 64 sequences, which keep their order, short sequences after long ones).
ROUNDS = [  # (contexts, query heads, KV heads, rows, layers, stale)
    ([16000, 8000, 8000, 8000], 4, 1, 16, 64, True),
    ([3072] * 8 + [100 + i % 29 for i in range(60)] + [2900] * 4, 8, 8, 5, 1, True),
    ([30000], 4, 1, 16, 100, True),  # whole teams, the last round not full
    ([300, 200, 40], 8, 8, 3, 200, False),  # a CTA per problem
]


@pytest.mark.parametrize("ctx,hq,hkv,n_q,layers,stale", ROUNDS)
def test_more_rounds_than_the_work_table(ctx, hq, hkv, n_q, layers, stale):
    case = make(ctx, hq, hkv, 128, n_q, 0, layers=layers)
    plan = binding.describe_plan(binding.WS_VERIFY, binding._kv_struct(case.kv), n_q, max(ctx))
    work = schedule(plan[1], plan[2], plan[5], ctx, layers * hkv)
    assert len(work[0]) > TABLE
    assert stale == any(mine[u][0] <= 1 and mine[u - TABLE][0] > 1 for mine in work for u in range(TABLE, len(mine)))
    for _ in range(2):  # the second pass finds the counters as the first one left them
        check(case, max(ctx))


def test_back_to_back_passes_are_bit_identical():
    """Nothing waits between the passes: partials, counters and score regions are used again by the next launch."""
    for ctx, hq, hkv, n_q in (([2061, 1571, 2799, 3337, 2804, 1373, 4224, 1213, 2610, 1552], 16, 2, 5),
                              ([851, 957, 1057, 1061, 1046, 1766], 16, 2, 8)):
        a, b = make(ctx, hq, hkv, 128, n_q, 0, seed=1), make(ctx, hq, hkv, 128, n_q, 0, seed=2)
        out, lse, stats, ws = check(a, max(ctx))
        want = out.clone(), stats.clone()
        for _ in range(25):
            binding.spec_verify_attn(b.kv, b.q_verify, b.ctx_len, max(ctx), out=out, lse=lse, stats=stats, workspace=ws)
            binding.spec_verify_attn(a.kv, a.q_verify, a.ctx_len, max(ctx), out=out, lse=lse, stats=stats, workspace=ws)
            torch.cuda.synchronize()
            assert torch.equal(out, want[0]) and torch.equal(stats, want[1])
        assert binding.read_status(ws) == 0


def test_two_rounds_on_fresh_tensors():
    """Two rounds per team at five tiles per CTA and four K/V slots: the second round's K tiles come a whole turn of the
    slot ring after the first one's V tiles, and the next K Q^T may start as soon as its score region is free."""
    ctx, T = [20000], 20000
    want = None
    for it in range(150):
        if it % 30 == 0:
            case = make(ctx, 32, 8, 128, 9, 0, seed=1)
        out, lse, stats, ws = binding.spec_verify_attn(case.kv, case.q_verify, case.ctx_len, T)
        torch.cuda.synchronize()
        assert binding.read_status(ws) == 0
        if want is None:
            want = out, lse, stats
            check(case, T)
        assert all(torch.equal(a, b) for a, b in zip((out, lse, stats), want))


def test_more_sequences_than_sixteen_bits_count():
    """65600 sequences of at most 16 tokens, one head: the last 64 are not their namesakes 65536 below."""
    B, n_q, D = 65600, 2, 64
    g = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()
    kv = inputs.KVCache(k=rand(1, B, 1, 16, D), v=rand(1, B, 1, 16, D), layer_stride=B * 16 * D, page_stride=16 * D,
                        head_stride=16 * D, slot_stride=D, n_layers=1, page_size=16, page_table=None, max_pages=1, batch=B,
                        n_q_heads=1, n_kv_heads=1, head_dim=D)
    q = rand(1, B, n_q, 1, D)
    lens = torch.randint(n_q, 17, (B,), generator=g, device="cuda", dtype=torch.int32)
    out, lse, stats, ws = binding.spec_verify_attn(kv, q, lens, 16)
    assert binding.read_status(ws) == 0 and binding.last_verify_impl() == binding.VERIFY_TCGEN05_CACHED
    s = torch.einsum("bqd,bkd->bqk", q[0, :, :, 0].double(), kv.k[0, :, 0].double()) / D ** 0.5
    last = lens[:, None].long() - n_q + torch.arange(n_q, device="cuda")
    s = s.masked_fill(torch.arange(16, device="cuda") > last[..., None], -float("inf"))
    p = s.softmax(-1)
    assert (out[0, :, :, 0].double() - p @ kv.v[0, :, 0].double()).abs().max().item() <= TOL
    assert (lse[0, :, :, 0].double() - s.logsumexp(-1)).abs().max().item() <= TOL
    seen = torch.arange(16, device="cuda") < lens[:, None]
    assert ((stats[0, :, 0, :16].double() - p.sum(1)) * seen).abs().max().item() <= TOL
