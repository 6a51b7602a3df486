"""Order of the Q-Mean key sums in the kernel with two query blocks per CTA (hifa4_attention_pair.cu): the slot of tile c is
filled again for tile c + 8, so every read of it has to happen before that load.  The kernel's waits and arrivals, restated as a
graph of events (an edge: happens before; the exchange of maxima, which differs between 64- and 128-key tiles, is left out: the
order must not need it).  The read has to be among the load's ancestors, for pairs of equal blocks, of blocks
that differ as a causal mask makes them differ, and of one block only."""
import random

import pytest

STAGES, SLOTS = 3, 8


def events(pairs, absent_waits=True):
    """pairs: (tiles of half 0, tiles of half 1) of the pairs one CTA takes.  Returns {event: events it waits for} and the halves
    that read tile c."""
    before, readers = {}, {}
    last = {}                                            # previous event of a thread or warp group, by name
    t = [0, 0]                                           # tiles of the half so far
    c0 = 0

    def add(ev, after=(), thread=None):
        deps = [e for e in after if e is not None]
        if thread is not None:
            if thread in last:
                deps.append(last[thread])
            last[thread] = ev
        before.setdefault(ev, []).extend(deps)

    for it, n in enumerate(pairs):
        n_max = max(n)
        for c in range(c0, c0 + n_max):                  # the loader moves on when the last V^T tile of the pair is on its way
            add(("load k", c), [("k free", h, c - STAGES) for h in (0, 1) if c >= STAGES], "loader k")
            add(("load v", c), [("v free", h, c - STAGES) for h in (0, 1) if c >= STAGES] + [("load k", c)], "loader v")
        for c in range(c0, c0 + n_max):
            if c == c0 and it > 0:
                before[("load k", c)].append(("load v", c0 - 1))
        for h in (0, 1):
            for jt in range(n_max):
                c, tt = c0 + jt, t[h] + jt
                if jt < n[h]:
                    add(("s", h, tt), [("load k", c), ("pull", h, tt - 1) if tt else None], ("issuer", h))
                    add(("k free", h, c), [("s", h, tt)])
                    g = ("softmax", h, tt % 2)
                    add(("pull", h, tt), [("s", h, tt)], g)
                    add(("read", h, tt), [("load k", c)], g)
                    readers.setdefault(c, []).append((h, tt))
                    add(("p", h, tt), [("pv", h, tt - 1) if jt else None], g)
                    add(("pv", h, tt), [("p", h, tt), ("load v", c), ("pv", h, tt - 1) if tt else None], ("issuer v", h))
                    add(("v free", h, c), [("pv", h, tt)])
                else:
                    wait = []
                    if n[h] == 0 and absent_waits:       # the half's softmax warps have reached this pair
                        wait = [last.get(("softmax", h, 0)), last.get(("softmax", h, 1))]
                    add(("k free", h, c), [("load k", c)] + wait, ("issuer", h))
                    add(("v free", h, c), [("load v", c)], ("issuer v", h))
            if n[h]:
                t[h] += n[h]
                for g in (0, 1):                         # output, after the block's last P V
                    add(("out", h, it, g), [("pv", h, t[h] - 1)], ("softmax", h, g))
        c0 += n_max
    return before, readers


def unordered(pairs, **kw):
    """Reads that are not ordered before the load that overwrites their slot."""
    before, readers = events(pairs, **kw)
    bad = []
    for c, who in readers.items():
        if ("load k", c + SLOTS) not in before:
            continue
        seen, todo = set(), [("load k", c + SLOTS)]
        while todo:
            e = todo.pop()
            for d in before.get(e, ()):
                if d not in seen:
                    seen.add(d)
                    todo.append(d)
        bad += [(c, h) for h, tt in who if ("read", h, tt) not in seen]
    return bad


def some_pairs(rng):
    def pair():
        n = rng.randint(1, 20)
        return rng.choice([(n, n), (n, 0), (n, max(1, n - 1)), (n, max(1, n - 2))])
    return [pair() for _ in range(rng.randint(2, 6))]


@pytest.mark.parametrize("seed", range(8))
def test_key_sums_are_read_before_their_slot_is_filled_again(seed):
    rng = random.Random(seed)
    for _ in range(40):
        pairs = some_pairs(rng)
        assert not unordered(pairs), pairs


def test_without_the_wait_of_an_absent_half_the_order_is_missing():
    assert unordered([(10, 10), (10, 0)], absent_waits=False)
    assert not unordered([(10, 10), (10, 10)], absent_waits=False)
