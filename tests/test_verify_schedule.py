"""The verification kernel's schedule and its work table, as a host model: every key tile of every problem is somebody's,
shares fit the score cache, and the rules by which the warps read the table never show one of them an entry
that is stale or overwritten.  The model's plans come from the library's own planner."""
import random

import pytest

from paper_2607_27735_b200 import binding
from test_plan_host import kv_struct
from verify_schedule import AHEAD, TABLE, schedule


def planned(lens, layers, hq, hkv, n_q, cap):
    plan = binding.describe_plan(binding.WS_VERIFY, kv_struct(layers, len(lens), hq, hkv, 128, cap), n_q, cap)
    assert plan[0] == 2
    return schedule(plan[1], plan[2], plan[5], lens, layers * hkv), plan


def draw(seed):
    rng = random.Random(seed)
    hkv = rng.choice([1, 2, 8])
    batch = rng.choice([1, 3, 8, 16, 64, 70, 100])
    layers = rng.choice([1, 4, 32]) if batch <= 16 else 1
    cap = rng.choice([768, 3072, 8064, 20096])  # whole tiles: the cache is one page per sequence
    lens = [max(20, int(cap * rng.random() ** rng.choice([1, 4]))) for _ in range(batch)]
    return lens, layers, hkv * rng.choice([1, 4]), hkv, rng.choice([2, 5, 9]), cap


@pytest.mark.parametrize("seed", range(60))
def test_every_tile_is_covered_once(seed):
    lens, layers, hq, hkv, n_q, cap = draw(seed)
    work, plan = planned(lens, layers, hq, hkv, n_q, cap)
    seen = {}
    for mine in work:
        for n, rank, b, head, t0, t1 in mine:
            if n:
                assert 0 < t1 - t0 <= plan[5]
                for t in range(t0, t1):
                    assert seen.setdefault((b, head, t), rank) == rank
                    seen[(b, head, t)] = rank
    assert len(seen) == sum((t + 127) // 128 for t in lens) * layers * hkv
    assert len({len(mine) for mine in work}) == 1


def walk(n_units, rng, reducer_obeys, publisher_waits):
    """Random interleavings of the publisher and the three warps that skip idle units; True if every read was right."""
    table, limit, at, pub = list(range(TABLE)), TABLE, [0, 0, 0], 0
    speed = [rng.choice([1, 30]) for _ in range(4)]
    while min(at) < n_units:
        who = rng.choices(range(4), weights=speed)[0]
        if who == 3:
            new = pub + AHEAD
            if pub >= n_units:
                continue
            if TABLE <= new < n_units:
                if publisher_waits and min(at) <= new - TABLE:
                    continue
                table[new % TABLE] = new
                limit = new + 1
            pub += 1
        elif at[who] < n_units and (at[who] < limit or (who == 2 and not reducer_obeys)):
            if table[at[who] % TABLE] != at[who]:
                return False
            at[who] += 1
    return True


def test_the_table_shows_every_warp_its_own_unit():
    rng = random.Random(1)
    assert all(walk(n, rng, True, True) for n in (1, 31, 32, 33, 40, 64, 200) for _ in range(50))
    # without the limit, or without the publisher's wait, some order of events shows a wrong entry
    assert not all(walk(64, rng, False, True) for _ in range(50))
    assert not all(walk(64, rng, True, False) for _ in range(50))
