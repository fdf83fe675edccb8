"""The ring of tile buffers of line_kernel (line_pass.cuh), modelled on the host:
which loads are under way when groups of threads give up.

The kernel's rules, restated: load q lands in buffer q mod NBUF and signals barrier
q mod 2 NBUF; the group that has read it for the last time issues load q + NBUF; a
group takes its loads in order (of OP_Z_DIV_SUM the three of a tile) and gives up
at the first whose wait runs out.  Before the CTA exits, every load that was
issued and not waited for must be among those that the kernel's last waits name,
and no other, and every wait must name its barrier's current phase."""

import random

import pytest


def last_waits(gr_n, per, nbuf, loads, stop):
    """The loads that the kernel waits for at its end (lane t < 4 GR)."""
    out = set()
    for t in range(4 * gr_n):
        g = t // 4
        if stop[g] < 0:
            continue
        n = stop[g] // (per * gr_n) * per + stop[g] % per + t % 4
        q = (n // per * gr_n + g) * per + n % per
        if q < loads and (q < nbuf or stop[(q - nbuf) // per % gr_n] < 0 or q - nbuf < stop[(q - nbuf) // per % gr_n]):
            out.add(q)
    return out


def run(gr_n, per, units, rng):
    nbuf, loads = gr_n + gr_n // 2, units * per
    own = [[q for i in range(g, units, gr_n) for q in range(i * per, (i + 1) * per)] for g in range(gr_n)]
    issued, consumed, stop, pos = set(range(min(nbuf, loads))), set(), [-1] * gr_n, [0] * gr_n
    live = set(range(gr_n))
    while live:
        g = rng.choice(sorted(live))
        if pos[g] == len(own[g]):
            live.discard(g)
            continue
        q = own[g][pos[g]]
        if q in issued and rng.random() > 0.04:
            # the wait names phase q // 2 NBUF by its parity: the phase before must be over, and its load this group's own
            assert q < 2 * nbuf or (q - 2 * nbuf in consumed and q - 2 * nbuf in own[g])
            consumed.add(q)
            pos[g] += 1
            if q + nbuf < loads:
                assert q + nbuf not in issued
                issued.add(q + nbuf)
        elif q in issued or all(own[h][pos[h]] not in issued for h in live if pos[h] < len(own[h])):
            stop[g] = q                               # its wait has run out, or nobody is left to issue its load
            live.discard(g)
    return issued - consumed, last_waits(gr_n, per, nbuf, loads, stop)


@pytest.mark.parametrize("groups", [2, 4, 8])
@pytest.mark.parametrize("per", [1, 3])
def test_loads_under_way_are_waited_for(groups, per):
    rng = random.Random(groups * 10 + per)
    gave_up = 0
    for units in (1, 2, 3, 5, 8, 13, 30):
        for _ in range(200):
            left, waited = run(groups, per, units, rng)
            gave_up += bool(left)
            assert left == waited
    assert gave_up > 100
