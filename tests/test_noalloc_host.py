"""Which shapes the entry point without a workspace takes (no GPU: a shape that is taken fails later, for want of a
device; nothing is launched and no pointer is read).  The measure is restated here: the status block, two counters per
problem and the partial results of the CTAs, dealt out evenly to a divisor of the KV heads, have to fit the built-in scratch
for either tensor-core kernel that can run, and the generic kernels' partials as well.  The split that the call then runs
with is another matter."""
import ctypes
import random

import pytest
import torch

from paper_2607_27735_b200 import binding
from test_plan_host import NSM, kv_struct

TOO_SMALL, SCRATCH = -3, 16 << 20
P = ctypes.c_void_p(1 << 20)

pytestmark = pytest.mark.skipif(torch.cuda.is_available(), reason="a taken shape would be launched")


def taken(kv, n_q, ctx):
    rc = binding.load().spec_verify_attn_noalloc(ctypes.byref(kv), P, n_q, P, ctx, 16, P, None, P, ctx, None)
    assert rc < 0
    return rc != TOO_SMALL


def up(x):
    return (x + 255) // 256 * 256


def heads_at_once(hkv, nb, tiles, score_less):
    best, pick = -1.0, 0
    for hg in range(1, hkv + 1):
        cph = NSM // hg
        if hkv % hg == 0 and cph and -(-nb // cph) <= tiles:
            score = nb * hg / (NSM * -(-nb // cph)) + 0.001 * hg - score_less(hg)
            if score > best:
                best, pick = score, hg
    return pick


def expected(layers, batch, hq, hkv, d, n_q, ctx):
    rows, nb, probs = n_q * hq // hkv, (ctx + 127) // 128, layers * batch * hkv
    n = (rows + 15) // 16 * 16
    splits = max(1, min(64, nb, (4 * 148 + probs - 1) // probs))
    generic = up(up(up(256 + probs * splits * rows * 8) + probs * rows * 4) + probs * splits * rows * d * 4)

    def partials(hg):
        ctas = hg * (NSM // hg)
        return up(up(up(256 + (2 * probs + 1) * 4) + 4 * ctas * rows * 8) + 4 * ctas * rows * 512)

    need = [generic]
    cached = heads_at_once(hkv, nb, min(32, (512 - 2 * n) // n), lambda hg: 0.0)
    assert cached  # (longer contexts run in two halves of the rows: not drawn here)
    need.append(partials(cached))
    if d == 128:
        need.append(partials(heads_at_once(hkv, nb, 1 << 30, lambda hg: (0.3 if hg * ctx * 256 / 2 ** 20 > 40 else 0.0) +
                                           (0.1 if layers * batch * (hkv // hg) < 2 else 0.0))))
    return max(need) <= SCRATCH


def test_counters_leave_the_partials_their_room():
    # 56 rows on 144 CTAs: 3840 bytes are left for counters
    assert taken(kv_struct(1, 1, 32, 8, 128, 2048), 14, 2048)
    assert taken(kv_struct(1, 1, 64, 16, 128, 2048), 14, 2048)


def test_the_split_does_not_decide():
    """Batches whose own split would put partials on all 148 CTAs, and groups whose even split leaves many of them out."""
    taken_at_56, rng = 0, random.Random(5)
    for _ in range(4000):
        hkv = rng.choice([1, 2, 4, 8, 16, 32])
        rows = rng.choice([20, 36, 50, 54, 55, 56, 57, 60, 62, 63, 64])
        g = rng.choice([x for x in range(1, 65) if rows % x == 0 and rows // x <= 32])
        layers, batch = rng.choice([1, 1, 2, 4]), rng.choice([1, 2, 4, 9, 30])
        d, ctx = rng.choice([64, 128]), rng.choice([128, 384, 1024, 2048, 4096, 8192, 16384])
        kv = kv_struct(layers, batch, g * hkv, hkv, d, ctx)
        want = expected(layers, batch, g * hkv, hkv, d, rows // g, ctx)
        assert taken(kv, rows // g, ctx) == want, (layers, batch, g, hkv, d, rows, ctx)
        taken_at_56 += want and rows > 54
    assert taken_at_56 > 50


def test_many_rows_are_refused():
    assert not taken(kv_struct(24, 1, 32, 8, 128, 4096), 16, 4096)  # 64 rows: 19 MB of partials
