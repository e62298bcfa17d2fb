"""What linking first pairs and leaving out z pairs saves, and the form of the cluster kernel: its
rows are cut into blocks wherever a CTA's share ends, links and dropped pairs stay inside a block,
and the pairs between blocks are united on their own.  On the CPU, word by word."""
import random

import pytest

from test_pair_rules import M, fill_down, fill_up, find, runs, starts


def rows(rng, p, n):
    return [sum((rng.random() < p) << x for x in range(32)) for _ in range(n)]


def number(w):
    base, total = [], 0
    for m in w:
        base.append(total)
        total += bin(starts(m)).count("1")
    return total, lambda r, x: base[r] + bin(starts(w[r]) & ((2 << x) - 1)).count("1") - 1


def unite(par, a, b):
    a, b = find(par, a), find(par, b)
    par[max(a, b)] = min(a, b)


def links_and_rest(w, r, my, mz, mzy):
    """Bits at which row r links, and at which its y and z pairs are left to unite."""
    m = w[r]
    oy, oz = m & my, m & mz
    uy = fill_up(m, oy)
    osy, osz = starts(oy), starts(oz)
    link = osy & ~(uy << 1) & M
    zlink = osz & ~(fill_up(m, oz) << 1) & ~(uy | fill_down(m, oy)) & M
    return link | zlink, osy & ~link, osz & ~zlink & ~(my & mzy)


@pytest.mark.parametrize("p,most", [(0.3116, 0.35), (0.5, 0.6)])
def test_few_unions_are_left(p, most):
    """A run starts at p (1 - p) of the sites and a pair of either kind at p^2 (1 - p^2), so 2 p (1 + p)
    pairs a run (0.82 at p_c, 1.5 at 1/2); less than half of them may be left."""
    rng = random.Random(12)
    total = rest = every = 0
    for _ in range(12):
        w = rows(rng, p, 16 * 16)
        total += number(w)[0]
        for r in range(len(w)):
            my, mz = (w[r - 1] if r % 16 else 0), (w[r - 16] if r >= 16 else 0)
            _, osy, osz = links_and_rest(w, r, my, mz, w[r - 17] if r % 16 and r >= 16 else 0)
            rest += bin(osy).count("1") + bin(osz).count("1")
            every += len(runs(w[r] & my)) + len(runs(w[r] & mz))
    assert rest < most * total and rest < every / 2


@pytest.mark.parametrize("p", [0.2, 0.3116, 0.6, 0.95])
@pytest.mark.parametrize("ny,nz,block", [(9, 7, 5), (9, 7, 13), (4, 16, 9), (16, 4, 24), (1, 20, 7), (7, 9, 63)])
def test_blocks_of_rows(ny, nz, block, p):
    rng = random.Random(ny * 100 + block)
    for _ in range(3):
        w = rows(rng, p, ny * nz)
        total, run = number(w)
        every, some = list(range(total)), list(range(total))
        for r, m in enumerate(w):
            for q, ok in ((r - 1, r % ny > 0), (r - ny, r >= ny)):
                for x in runs(m & w[q]) if ok else []:
                    unite(every, run(r, x), run(q, x))
        rest, cross = [], []
        for r, m in enumerate(w):
            ls, y, z = r % block, r % ny, r // ny           # place in its block
            iny, inz = y > 0 and ls >= 1, z > 0 and ls >= ny
            my, mz = (w[r - 1] if iny else 0), (w[r - ny] if inz else 0)
            mzy = w[r - ny - 1] if my and mz and ls >= ny + 1 else 0
            link, osy, osz = links_and_rest(w, r, my, mz, mzy)
            for x in range(32):
                if (link >> x) & 1:
                    q = r - 1 if (my >> x) & 1 else r - ny
                    assert some[run(r, x)] == run(r, x) and run(q, x) < run(r, x) and q // block == r // block
                    some[run(r, x)] = run(q, x)
                if (osy >> x) & 1:
                    rest.append((run(r, x), run(r - 1, x)))
                if (osz >> x) & 1:
                    rest.append((run(r, x), run(r - ny, x)))
            if y > 0 and not iny:
                cross += [(run(r, x), run(r - 1, x)) for x in runs(m & w[r - 1])]
            if z > 0 and not inz:
                cross += [(run(r, x), run(r - ny, x)) for x in runs(m & w[r - ny])]
        for a, b in rest + cross:
            unite(some, a, b)
        assert [find(every, i) for i in range(total)] == [find(some, i) for i in range(total)]
