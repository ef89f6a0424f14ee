"""The hand-off between softmax, correction warps and accumulator issuer of the pipelined attention
kernels (vc_attn_fwd_2q.cuh, vc_attn_fwd4.cu), restated as a state machine on mbarriers and explored
over every order of events: no product runs while a row's accumulator is being rescaled, no arrival
counts for another key tile's phase, nobody waits for a phase that has gone by.

One query tile of the kernels: the softmax warpgroup (its threads advance together here), two
correction warps - the maxima of one never move, those of the other move at every key tile or at any
subset of them - and the issuer, whose products complete some time after they were issued."""
import itertools

import pytest


class Bar:
    """An mbarrier: a phase completes when `count` arrivals are in; a wait by parity passes while the
    current phase's parity differs from the one asked for."""
    def __init__(self, count):
        self.count = count


def explore(two, smooth, nb, moved_at, slots, last_wait_first):
    """First fault found, or None.  State: program counters of the four agents, barrier phases and pending
    arrivals, products issued and completed.

    two: pairs of query tiles (products alternate on one o_done barrier per tile), else one tile with two.
    slots: pc_full barriers a tile's hand-offs alternate between.  last_wait_first: without block means the wait
    for the last product but one on the last product's barrier stands in front of the last arrival, not behind it."""
    n_od = 1 if two else 2                       # o_done barriers
    n_a = 2 if two else 4                        # alpha barriers and slots
    counts = {("pc", i): 4 for i in range(slots)}
    counts.update({("a", i): 1 for i in range(n_a)})
    counts.update({("od", i): 1 for i in range(n_od)})

    def pc(j): return ("pc", j % slots), (j // slots) & 1
    def al(j): return ("a", j % n_a), (j // n_a) & 1
    def od(j): return ("od", j % n_od), (j // n_od) & 1

    def softmax():
        prog = []
        for j in range(nb):
            prog += [("arrive", al(j)[0], 1, j)]
            if j - n_od >= 0:
                prog += [("wait", *od(j - n_od))]
            prog += [("arrive", pc(j)[0], 2, j)]
        return prog

    def correction(moves):
        prog = []
        before = n_od                            # tiles between products on one barrier
        for j in range(nb):
            prog += [("wait", *al(j))]
            if j > 0 and (smooth or j in moves):
                prog += [("wait", *od(j - 1))]
                if j in moves:
                    prog += [("begin", j), ("end", j)]
            if not smooth and last_wait_first and j == nb - 1 and j - before >= 0:
                prog += [("wait", *od(j - before))]
            prog += [("arrive", pc(j)[0], 1, j)]
        if not smooth and not last_wait_first and nb - 1 - before >= 0:
            prog += [("wait", *od(nb - 1 - before))]
        return prog + [("wait", *od(nb - 1)), ("read", nb - 1)]

    def issuer():
        prog = []
        for j in range(nb):
            prog += [("wait", *pc(j)), ("issue", j)]
        return prog

    progs = [softmax(), correction(()), correction(moved_at), issuer()]
    names = sorted(counts)
    at = {n: i for i, n in enumerate(names)}
    # state: pcs, (phase, pending) per barrier, issued, completed, tile being rescaled (-1: none)
    start = ((0,) * 4, tuple((0, counts[n]) for n in names), 0, 0, -1)
    seen, todo = {start}, [start]

    def arrive(bars, name, n):
        bars = list(bars)
        phase, left = bars[at[name]]
        left -= n
        assert left >= 0
        bars[at[name]] = (phase + 1, counts[name]) if left == 0 else (phase, left)
        return tuple(bars)

    while todo:
        state = todo.pop()
        pcs, bars, issued, done, busy = state
        nxt = []
        if done < issued:                        # the oldest product completes
            nxt.append((pcs, arrive(bars, od(done)[0], 1), issued, done + 1, busy))
        for w, prog in enumerate(progs):
            if pcs[w] == len(prog):
                continue
            op = prog[pcs[w]]
            step = tuple(p + (i == w) for i, p in enumerate(pcs))
            if op[0] == "wait":
                if bars[at[op[1]]][0] & 1 != op[2]:
                    nxt.append((step, bars, issued, done, busy))
            elif op[0] == "arrive":
                name, n, j = op[1:]
                own = j // (slots if name[0] == "pc" else n_a)
                if bars[at[name]][0] != own:
                    return f"an arrival for key tile {j} counts for another phase"
                if bars[at[name]][1] < n:
                    return f"more arrivals than the phase of key tile {j} has room for"
                nxt.append((step, arrive(bars, name, n), issued, done, busy))
            elif op[0] == "issue":
                if busy >= 0:
                    return f"product {op[1]} issued while the rescale of key tile {busy} runs"
                nxt.append((step, bars, op[1] + 1, done, busy))
            elif op[0] == "begin":
                if done < issued or issued != op[1]:
                    return f"rescale of key tile {op[1]} with products {done} to {issued} in flight"
                nxt.append((step, bars, issued, done, op[1]))
            elif op[0] == "end":
                nxt.append((step, bars, issued, done, -1))
            else:
                if done != nb:
                    return f"accumulator read after {done} of {nb} products"
                nxt.append((step, bars, issued, done, busy))
        if not nxt and any(p < len(prog) for p, prog in zip(pcs, progs)):
            return "a wait that nothing ends: " + str([prog[p] for p, prog in zip(pcs, progs) if p < len(prog)])
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


def every_subset(nb):
    return itertools.chain.from_iterable(itertools.combinations(range(1, nb), r) for r in range(nb))


@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("two", [True, False])
def test_every_order_of_events_is_sound(two, smooth):
    for nb in range(1, 8):
        for moved in every_subset(nb):
            for slots in (2, 4) if smooth and not two else (2 if two else 4,):
                assert explore(two, smooth, nb, moved, slots, True) is None, (nb, moved, slots)


def test_two_barriers_do_not_serve_one_tile():
    """With one query tile and no block means a warp may be two key tiles ahead of another (with block means it may not)."""
    assert "another phase" in explore(False, False, 6, (2,), 2, True)


@pytest.mark.parametrize("two", [True, False])
def test_the_last_wait_stands_in_front_of_the_last_arrival(two):
    assert "a wait that nothing ends" in explore(two, False, 5, (), 2 if two else 4, False)
