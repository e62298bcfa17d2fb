"""The tile pass's word arithmetic against plain definitions, on the CPU: spreading bits
inside runs, and which run pairs need a union.  A run's first pair (with row y - 1, or
with row z - 1 if it meets no run of row y - 1) becomes a link, a z pair starting where the
sites at y - 1 are occupied on both planes is dropped, and the links and the rest must
join exactly the runs that all pairs join."""
import random

import pytest

M = 0xFFFFFFFF


def starts(m):
    return m & ~(m << 1) & M


def rev(v):
    return int(f"{v:032b}"[::-1], 2)


def fill_up(m, o):
    return ((((m + o) & M) ^ m) | o) & m


def fill_down(m, o):
    return rev(fill_up(rev(m), rev(o)))


def runs(m):
    return [x for x in range(32) if (starts(m) >> x) & 1]


def words(rng, n):
    special = [0, M, 1, 1 << 31, 0x55555555, 0xAAAAAAAA, 0x7FFFFFFE, 0x80000001]
    return special + [rng.getrandbits(32) | (rng.getrandbits(32) if k % 2 else 0) for k in range(n)]


def test_fills():
    rng = random.Random(4)
    ws = words(rng, 300)
    for m in ws:
        for c in rng.sample(ws, 40):
            o = c & m
            up = down = 0
            for s in runs(m):
                e = s
                while e < 31 and (m >> (e + 1)) & 1:
                    e += 1
                hit = [x for x in range(s, e + 1) if (o >> x) & 1]
                for x in range(s, e + 1):
                    up |= (1 << x) if hit and x >= hit[0] else 0
                    down |= (1 << x) if hit and x <= hit[-1] else 0
            assert fill_up(m, o) == up and fill_down(m, o) == down, (hex(m), hex(o))


def find(par, a):
    while par[a] != a:
        a = par[a]
    return a


@pytest.mark.parametrize("p", [0.1, 0.3116, 0.5, 0.8, 0.97, None])
@pytest.mark.parametrize("ty,tz", [(8, 8), (16, 3), (3, 16)])
def test_links_and_rest_join_what_all_pairs_join(p, ty, tz):
    rng = random.Random(hash((p, ty, tz)) & 0xffff)
    for _ in range(12):
        if p is None:
            w = [rng.choice(words(rng, 4)) for _ in range(ty * tz)]
        else:
            w = [sum((rng.random() < p) << x for x in range(32)) for _ in range(ty * tz)]
        base, total = [], 0
        for m in w:
            base.append(total)
            total += bin(starts(m)).count("1")

        def run(r, x):
            return base[r] + bin(starts(w[r]) & ((2 << x) - 1)).count("1") - 1

        every, some = list(range(total)), list(range(total))
        n_some = n_all = 0

        def unite(par, a, b):
            a, b = find(par, a), find(par, b)
            par[max(a, b)] = min(a, b)

        for r, m in enumerate(w):   # all pairs
            for q, ok in ((r - 1, r % ty > 0), (r - ty, r >= ty)):
                for x in runs(m & w[q]) if ok else []:
                    unite(every, run(r, x), run(q, x))
                    n_all += 1
        rest = []
        for r, m in enumerate(w):
            my, mz = (w[r - 1] if r % ty else 0), (w[r - ty] if r >= ty else 0)
            oy, oz = m & my, m & mz
            uy = fill_up(m, oy)
            osy, osz = starts(oy), starts(oz)
            link = osy & ~(uy << 1) & M
            osy ^= link
            zlink = osz & ~(fill_up(m, oz) << 1) & ~(uy | fill_down(m, oy)) & M
            link |= zlink
            osz &= ~zlink
            if r % ty and r >= ty:
                osz &= ~(my & w[r - ty - 1])
            for x in range(32):
                if (link >> x) & 1:
                    q = r - 1 if (my >> x) & 1 else r - ty
                    assert some[run(r, x)] == run(r, x) and run(q, x) < run(r, x)   # one link a run
                    some[run(r, x)] = run(q, x)
                if (osy >> x) & 1:
                    rest.append((run(r, x), run(r - 1, x)))
                if (osz >> x) & 1:
                    rest.append((run(r, x), run(r - ty, x)))
        for a, b in rest:
            unite(some, a, b)
        assert [find(every, i) for i in range(total)] == [find(some, i) for i in range(total)]
        assert len(rest) <= n_all
