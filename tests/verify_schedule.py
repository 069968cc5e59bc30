"""Host restatement of the verification kernel's schedule: which problem every CTA works on in every unit, from the plan
(``describe_plan``: teams, CTAs per team, score tiles a CTA holds) and the sequence lengths."""
SORT_MAX, MAX_CLASS, TILE = 64, 4, 128
TABLE, AHEAD = 32, 24  # units the work table holds, units the publisher warp writes ahead


def schedule(teams, cph, n_cache, lens, heads):
    """``heads`` = layers * KV heads.  Returns ``work[cta][unit] = (n, rank, sequence, head, t0, t1)``, n = 0: idle."""
    size = [cph >> f for f in range(MAX_CLASS) if cph >> f >= 1]
    subs = [cph // s for s in size]
    tiles = [(t + TILE - 1) // TILE for t in lens]
    order, count = list(range(len(lens))), [0] * len(size)
    if len(lens) > SORT_MAX:  # order kept, whole teams
        count[0] = len(lens)
    else:
        order.sort(key=lambda b: (-lens[b], b))
        for b in order:
            f = len(size) - 1
            while f > 0 and size[f] * n_cache < tiles[b]:
                f -= 1
            count[f] += 1
        for f in range(len(size) - 1, 0, -1):  # a class that would not fill half of a round joins the coarser one
            if 2 * count[f] * heads <= teams * subs[f]:
                count[f - 1] += count[f]
                count[f] = 0
    work = [[] for _ in range(teams * cph)]
    first = unit = 0
    for f in range(len(size)):
        slots = teams * subs[f]
        for u in range((count[f] * heads + slots - 1) // slots):
            for cta, mine in enumerate(work):
                team, local = divmod(cta, cph)
                sub, rank = divmod(local, size[f])
                slot = team * subs[f] + sub
                i = u * slots + (slots - 1 - slot if unit & 1 else slot)
                seq, head = divmod(i, heads)
                if sub >= subs[f] or seq >= count[f]:
                    mine.append((0, 0, 0, 0, 0, 0))
                    continue
                b = order[first + seq]
                n = min(size[f], tiles[b])
                if rank >= n:
                    mine.append((0, 0, 0, 0, 0, 0))
                else:
                    share = (lambda r: r) if n < size[f] else (lambda r: r * tiles[b] // size[f])
                    mine.append((n, rank, b, head, share(rank), share(rank + 1)))
            unit += 1
        first += count[f]
    return work
