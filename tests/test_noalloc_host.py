"""Which shapes the entry point without a workspace takes (no GPU: a shape that is taken fails later, for want of a
device; nothing is launched and no pointer is read)."""
import ctypes

import pytest
import torch

from paper_2607_27735_b200 import binding
from test_plan_host import kv_struct

TOO_SMALL = -3
P = ctypes.c_void_p(1 << 20)

pytestmark = pytest.mark.skipif(torch.cuda.is_available(), reason="a taken shape would be launched")


def taken(kv, n_q, ctx):
    rc = binding.load().spec_verify_attn_noalloc(ctypes.byref(kv), P, n_q, P, ctx, 16, P, None, P, ctx, None)
    assert rc < 0
    return rc != TOO_SMALL


def test_counters_leave_the_partials_their_room():
    # 56 rows on 144 CTAs: 3840 bytes are left for counters
    assert taken(kv_struct(1, 1, 32, 8, 128, 2048), 14, 2048)
    assert taken(kv_struct(1, 1, 64, 16, 128, 2048), 14, 2048)


def test_many_rows_are_refused():
    assert not taken(kv_struct(24, 1, 32, 8, 128, 4096), 16, 4096)  # 64 rows: 19 MB of partials
