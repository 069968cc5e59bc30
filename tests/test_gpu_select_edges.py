"""Selection at the edges of its forms: spans at and around the dense list's length and a sweep trip, rows that do not
start on 16 bytes, flat scores, scores whose large values sit in one stretch or only between the sample's blocks, zeros,
hundreds of equal scores at the threshold.  Integer work: bit-exact against the oracle."""
import pytest
import torch

import oracle
from paper_2607_27735_b200 import binding

pytestmark = pytest.mark.gpu


def check(stats, sel_len, k_sink, k_recent, k_total):
    idx, n = binding.spec_select_recall(stats, sel_len, k_sink, k_recent, k_total)
    r_idx, r_n = oracle.select_recall(stats.cpu(), sel_len.cpu(), k_sink, k_recent, k_total)
    assert torch.equal(idx.cpu(), r_idx) and torch.equal(n.cpu(), r_n)


# span = T - 68: 4096 is the longest dense one at a small budget, 8192 scores are a trip of the sweep
@pytest.mark.parametrize("span", [510, 4095, 4096, 4097, 8192, 8195, 20477, 20480, 40961])
@pytest.mark.parametrize("keep", [3, 400, "half"])
def test_spans_and_unaligned_rows(span, keep):
    g = torch.Generator(device="cuda").manual_seed(span)
    T = span + 68
    k_mid = span // 2 if keep == "half" else keep
    stats = torch.randn(1, 2, 3, T + 5, generator=g, device="cuda").exp_()  # row starts cycle through all alignments
    sel_len = torch.tensor([T, T - 1], dtype=torch.int32, device="cuda")
    check(stats, sel_len, 4, 64, k_mid + 68)


@pytest.mark.parametrize("T", [6000, 33333])
@pytest.mark.parametrize("kind", ["flat", "one_stretch", "between_samples", "zeros", "ties"])
def test_distributions(T, kind):
    g = torch.Generator(device="cuda").manual_seed(T)
    stats = torch.rand(1, 2, 2, T, generator=g, device="cuda")
    if kind == "flat":
        stats = 0.5 + 1e-5 * stats
    elif kind == "one_stretch":
        stats[..., T // 3:T // 3 + 1500] += 10.0
    elif kind == "between_samples":  # a sample of every fourth vector of a stretch of 16 sees none of the large ones
        big = torch.zeros(T, dtype=torch.bool, device="cuda")
        big[68:] = (torch.arange(T - 68, device="cuda") * 256 // (T - 68)) % 7 == 3
        stats = torch.where(big, stats + 10.0, stats)
    elif kind == "zeros":
        stats = torch.where(stats > 0.99, stats, torch.zeros_like(stats))
    else:
        kth = stats[..., 4:T - 71].topk(932, dim=-1).values[..., -1:]
        where = torch.rand(1, 2, 2, T, generator=g, device="cuda").argsort(dim=-1)[..., :700]
        stats.scatter_(-1, where, kth.expand(1, 2, 2, 700).contiguous())
    sel_len = torch.tensor([T, T - 7], dtype=torch.int32, device="cuda")
    check(stats.contiguous(), sel_len, 4, 64, 1000)


@pytest.mark.parametrize("T", [3000, 9000, 33333, 140000])
@pytest.mark.parametrize("kind", ["any", "some_negative", "nan", "minus_zero"])
def test_any_bit_pattern_is_ordered_as_an_unsigned_number(T, kind):
    """Scores are sums of probabilities; what else may lie in the buffer changes nothing but the order."""
    g = torch.Generator(device="cuda").manual_seed(T)
    n = (1, 1, 2, T)
    bits = torch.rand(n, generator=g, device="cuda").view(torch.int32)
    odd = {"any": torch.randint(-2 ** 31, 2 ** 31, n, generator=g, device="cuda", dtype=torch.int64).int(),
           "some_negative": (-torch.rand(n, generator=g, device="cuda")).view(torch.int32),
           "nan": torch.full(n, -1, dtype=torch.int32, device="cuda"),
           "minus_zero": torch.full(n, -2 ** 31, dtype=torch.int32, device="cuda")}[kind]
    share = 1.0 if kind == "any" else 0.03
    bits = torch.where(torch.rand(n, generator=g, device="cuda") < share, odd, bits)
    sel_len = torch.tensor([T], dtype=torch.int32, device="cuda")
    idx, cnt = binding.spec_select_recall(bits.view(torch.float32), sel_len, 4, 64, 1000)
    order = (bits.long() & 0xFFFFFFFF)[..., 4:T - 64] * 2 ** 18 + torch.arange(T - 68, 0, -1, device="cuda")
    mid = order.topk(932, dim=-1).indices.sort(dim=-1).values + 4
    want = torch.cat([torch.arange(4, device="cuda").expand(1, 1, 2, 4), mid,
                      torch.arange(T - 64, T, device="cuda").expand(1, 1, 2, 64)], dim=-1).int()
    assert torch.equal(idx, want) and bool((cnt == 1000).all())


# the position bitmap holds 131072 positions: spans that end around a multiple of it, large scores in one window only, equal
# scores at the threshold in all of them, and lengths whose sample grows
@pytest.mark.parametrize("T,k_total", [(131072 + 63, 1024), (131072 + 64, 1024), (131072 + 65, 4096), (262144 + 64, 4096),
                                       (262144 + 65, 2048), (300001, 4096), (1048576 + 4, 4096), (3000001, 4096)])
@pytest.mark.parametrize("where", ["anywhere", "first", "last", "ties", "flat", "zeros"])
def test_contexts_of_several_windows(T, k_total, where):
    g = torch.Generator(device="cuda").manual_seed(T)
    stats = torch.rand(1, 1, 2, T, generator=g, device="cuda") ** 8
    if where in ("first", "last"):
        stats[..., slice(4, 5000) if where == "first" else slice(T - 5064, T - 64)] += 1.0
    elif where == "ties":
        tie = torch.rand(1, 1, 2, T, generator=g, device="cuda") < 1.2 * k_total / T
        stats = torch.where(tie, torch.full_like(stats, 0.999), 0.99 * stats)
    elif where == "flat":
        stats = 0.5 + 1e-5 * stats
    elif where == "zeros":  # fewer positive scores than the budget takes
        few = torch.rand(1, 1, 2, T, generator=g, device="cuda") < 0.3 * k_total / T
        stats = torch.where(few, stats + 1e-3, torch.zeros_like(stats))
    check(stats.contiguous(), torch.tensor([T], dtype=torch.int32, device="cuda"), 4, 64, k_total)


@pytest.mark.parametrize("n_equal", [512, 513, 2000])
@pytest.mark.parametrize("T", [3000, 9000, 33333])
def test_the_lowest_of_equal_scores(T, n_equal):
    """The threshold among n_equal equal scores, up to which the pairwise ranking goes or does not."""
    g = torch.Generator(device="cuda").manual_seed(T + n_equal)
    stats = torch.rand(1, 1, 3, T, generator=g, device="cuda") * 0.5
    at = torch.rand(1, 1, 3, T, generator=g, device="cuda").argsort(dim=-1)
    stats.scatter_(-1, at[..., :n_equal], 0.75)
    stats.scatter_(-1, at[..., n_equal:n_equal + 300], 0.9)
    check(stats, torch.tensor([T], dtype=torch.int32, device="cuda"), 4, 64, 800)
