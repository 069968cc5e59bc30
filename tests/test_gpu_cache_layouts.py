"""Verification over the same keys and values laid out in memory in different ways: what the copies of whole rows are built from
is the strides' greatest common divisor, so heads outside pages, heads between rows, padded rows, layers inside
pages and pages of 8 to 256 tokens have to give the bits that the dense order gives, and whole rows those of the halves (the
arithmetic behind the copies is the same)."""
import dataclasses

import pytest
import torch

import oracle
from paper_2607_27735_b200 import binding, inputs

pytestmark = pytest.mark.gpu
TOL = 2e-3
L, H, D, N_Q = 2, 2, 128, 5


def laid_out(kv, order, pad):
    """``kv`` ([layer, page, head, slot, D]) with its first four axes stored in ``order`` and ``pad`` elements behind each row."""
    axes = [kv.n_layers, kv.k.shape[1], kv.n_kv_heads, kv.page_size]
    strides, step = [0] * 4, D + pad
    for a in reversed(order):
        strides[a] = step
        step *= axes[a]
    def store(x):
        flat = torch.full((step + D,), 7.0, device=x.device, dtype=x.dtype)
        flat.as_strided(axes + [D], strides + [1]).copy_(x)
        return flat
    return dataclasses.replace(kv, k=store(kv.k), v=store(kv.v), layer_stride=strides[0], page_stride=strides[1],
                               head_stride=strides[2], slot_stride=strides[3], n_pages=kv.k.shape[1])


def poison(case, ctx):
    """NaN in every slot behind a sequence's context (in the pages the table gives it)."""
    kv = case.kv
    for b, t in enumerate(ctx):
        for page in range(kv.max_pages):
            first = max(0, t - page * kv.page_size)
            if first < kv.page_size:
                kv.k[:, kv.phys_page(b, page), :, first:] = float("nan")
                kv.v[:, kv.phys_page(b, page), :, first:] = float("nan")


# pages of up to 64 tokens are copied as whole rows, larger ones as halves, those above 128 in pieces
@pytest.mark.parametrize("page", [8, 16, 64, 128, 256])
@pytest.mark.parametrize("ctx", [[700, 129, 128], [9]])
def test_every_order_gives_the_bits_of_the_dense_one(page, ctx):
    cfg = inputs.small_config(ctx=(min(ctx), max(ctx)), n_q=N_Q, n_q_heads=4 * H, n_kv_heads=H, head_dim=D, planted=4,
                              batch=len(ctx), n_layers=L, page_size=page, shuffled_pages=True, seed=5)
    case = inputs.make_case(cfg, device="cuda", ctx_override=ctx)
    T = max(ctx)
    poison(case, ctx)
    ref = binding.spec_verify_attn(case.kv, case.q_verify, case.ctx_len, T)
    assert binding.read_status(ref[3]) == 0
    o_out, o_lse, o_stats = oracle.verify_attn(case.kv.cpu(), case.q_verify.cpu(), case.ctx_len.cpu(), 16, ref[2].shape[-1])
    for got, want in zip(ref, (o_out, o_lse, o_stats)):
        assert (got.cpu().double() - want).abs().max().item() <= TOL
    for order, pad in (((0, 1, 2, 3), 8), ((0, 1, 3, 2), 0), ((2, 0, 1, 3), 0), ((1, 0, 2, 3), 24), ((3, 2, 1, 0), 0), ((0, 2, 1, 3), 8)):
        out, lse, stats, ws = binding.spec_verify_attn(laid_out(case.kv, order, pad), case.q_verify, case.ctx_len, T)
        assert binding.read_status(ws) == 0
        assert torch.equal(out, ref[0]) and torch.equal(lse, ref[1])
        for b, t in enumerate(ctx):
            assert torch.equal(stats[:, b, :, :t], ref[2][:, b, :, :t])


def test_rows_beyond_31_bits_take_the_other_map():
    """A pool whose rows cannot be numbered in 31 bits (it is only said to be that large; the pages in use are the same): tiles
    are copied half by half into the other layout, which gives the same bits."""
    cfg = inputs.small_config(ctx=(700, 700), n_q=N_Q, n_q_heads=4 * H, n_kv_heads=H, head_dim=D, planted=4, n_layers=L,
                              page_size=16, shuffled_pages=True, seed=6)
    case = inputs.make_case(cfg, device="cuda")
    poison(case, [700])
    ref = binding.spec_verify_attn(case.kv, case.q_verify, case.ctx_len, 700)
    assert torch.isfinite(ref[0]).all()
    large = dataclasses.replace(case.kv, n_pages=(1 << 30) + 8)
    out, lse, stats, ws = binding.spec_verify_attn(large, case.q_verify, case.ctx_len, 700)
    assert binding.read_status(ws) == 0
    assert torch.equal(out, ref[0]) and torch.equal(lse, ref[1]) and torch.equal(stats[..., :700], ref[2][..., :700])


# Rows per KV head that fill one, two, three and four warpgroups of different widths (8, 20, 36, 64, 68, 96, 104 and 128
# rows are the eight widths of the score columns), each statistic, and tiles as whole rows and as halves (a pool that is
# said to be too large to number its rows takes the halves).
# Pages of 64 tokens and of 16 are the largest that are copied as whole rows, up to 64 rows and above.
@pytest.mark.parametrize("n_q,kind,page", [(2, "sum", 16), (5, "per_head", 64), (9, "group_max", 16), (12, "sum", 64), (13, "sum", 64),
                                           (13, "per_head", 16), (16, "hist", 32), (17, "sum", 16), (17, "per_head", 16), (24, "sum", 16),
                                           (26, "group_max", 16), (32, "hist", 16), (32, "sum", 32)])
def test_rows_and_statistics_in_both_tile_layouts(n_q, kind, page):
    group = 4
    ctx = [700, 33, 135]
    cfg = inputs.small_config(ctx=(min(ctx), max(ctx)), n_q=n_q, n_q_heads=group * H, n_kv_heads=H, head_dim=D, planted=4, batch=len(ctx),
                              n_layers=L, page_size=page, shuffled_pages=True, seed=7)
    case = inputs.make_case(cfg, device="cuda", ctx_override=ctx)
    o_out, o_lse, o_stats = oracle.verify_attn(case.kv.cpu(), case.q_verify.cpu(), case.ctx_len.cpu(), 16, 704,
                                               per_head=kind == "per_head", group_max=kind == "group_max")
    poison(case, ctx)
    heads = group * H if kind == "per_head" else H

    def call(kv):
        hist = torch.zeros(L, len(ctx), heads, 2048, dtype=torch.int32, device="cuda") if kind == "hist" else None
        out, lse, stats, ws = binding.spec_verify_attn(kv, case.q_verify, case.ctx_len, 700, per_head=kind == "per_head",
                                                       group_max=kind == "group_max", score_hist=hist)
        assert binding.read_status(ws) == 0 and binding.last_verify_impl() == binding.VERIFY_TCGEN05_CACHED
        return out, lse, stats, hist

    ref = call(case.kv)
    assert (ref[0].cpu().double() - o_out).abs().max().item() <= TOL
    assert (ref[1].cpu().double() - o_lse).abs().max().item() <= TOL
    assert (ref[2].cpu().double() - o_stats).abs().max().item() <= TOL
    for kv in (dataclasses.replace(case.kv, n_pages=(1 << 30) + 8), laid_out(case.kv, (2, 0, 1, 3), 8), laid_out(case.kv, (0, 1, 3, 2), 0)):
        got = call(kv)
        for a, b in zip(ref, got):
            assert a is None or torch.equal(a, b)


def test_rows_in_two_passes_in_another_order_of_the_axes():
    """68 rows at a context whose share of keys does not fit the score cache: two passes, each over both layouts."""
    T = 80000
    cfg = inputs.small_config(ctx=(T, T), n_q=17, n_q_heads=8, n_kv_heads=2, head_dim=D, planted=4, n_layers=1, page_size=16,
                              shuffled_pages=True, seed=8)
    case = inputs.make_case(cfg, device="cuda")
    poison(case, [T])
    got = []
    for kv in (case.kv, dataclasses.replace(case.kv, n_pages=(1 << 30) + 8), laid_out(case.kv, (0, 3, 1, 2), 8)):
        out, lse, stats, ws = binding.spec_verify_attn(kv, case.q_verify, case.ctx_len, T)
        assert binding.read_status(ws) == 0 and binding.last_verify_impl() == binding.VERIFY_TCGEN05_CACHED_2PASS
        assert torch.isfinite(out).all()
        got.append((out, lse, stats))
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0], other))


# A stride of 0 over an extent above 1: every head, page or layer the same rows.  Each of the maps that copies are built from
# has to read it so: whole rows, halves (128-token pages, head_dim 64, a pool too large to number its rows), bytes, two sweeps.
@pytest.mark.parametrize("axis", ["layer", "page", "head"])
@pytest.mark.parametrize("what", ["rows", "halves", "dim64", "large", "fp8", "fp8_dim64", "two_sweeps"])
def test_an_axis_of_stride_zero_is_a_broadcast(axis, what):
    ctx = [400, 129]
    dim, page = (64 if "dim64" in what else D), (128 if what == "halves" else 16)
    cfg = inputs.small_config(ctx=(min(ctx), max(ctx)), n_q=N_Q, n_q_heads=4 * H, n_kv_heads=H, head_dim=dim, planted=4, batch=len(ctx),
                              n_layers=L, page_size=page, shuffled_pages=True, seed=9)
    case = inputs.make_case(cfg, device="cuda", ctx_override=ctx)
    kv = case.kv
    if what.startswith("fp8"):
        kv = inputs.quantize_kv_fp8(kv)
        # other scales per head and layer, within a factor of 1.5 of the quantisation's: values stay of the order of 1 (up to 7),
        # which TOL is stated for (it is absolute; probabilities carry 2^-14 and fp32 sums of them)
        kv = dataclasses.replace(kv, k_scale=kv.k_scale * (torch.rand_like(kv.k_scale) + 0.5),
                                 v_scale=kv.v_scale * (torch.rand_like(kv.v_scale) + 0.5))
    at = {"layer": 0, "page": 1, "head": 2}[axis]
    def spread(x):  # the same rows written out for every place of the axis
        x = x.clone()
        x.copy_(x.select(at, 0).unsqueeze(at).expand_as(x))
        return x
    dense = dataclasses.replace(kv, k=spread(kv.k), v=spread(kv.v))
    zero = dataclasses.replace(kv, **{axis + "_stride": 0})
    if what == "large":
        zero = dataclasses.replace(zero, n_pages=(1 << 30) + 8)
    prev = binding.set_verify_impl(binding.VERIFY_TCGEN05_TWOSWEEP if what == "two_sweeps" else binding.VERIFY_AUTO)
    try:
        ref = binding.spec_verify_attn(dense, case.q_verify, case.ctx_len, max(ctx))
        got = binding.spec_verify_attn(zero, case.q_verify, case.ctx_len, max(ctx))
    finally:
        binding.set_verify_impl(prev)
    assert binding.read_status(ref[3]) == 0 and binding.read_status(got[3]) == 0
    o_out, o_lse, o_stats = oracle.verify_attn(dense.cpu(), case.q_verify.cpu(), case.ctx_len.cpu(), 16, ref[2].shape[-1])
    for a, b, o in zip(ref, got, (o_out, o_lse, o_stats)):
        assert (a.cpu().double() - o).abs().max().item() <= TOL
        assert (b.cpu().double() - o).abs().max().item() <= TOL
