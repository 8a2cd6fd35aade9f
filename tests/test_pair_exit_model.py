"""Host-side model of the barriers of a CTA pair (linear_pair_kernel in csrc/w4a8_linear_pair.cuh).  The kernel's closing cluster
barrier orders execution only, so everything that one CTA sends into the other's shared memory -- arrivals of its warps,
commits of the leader's tensor cores, bytes of its activation tiles -- must have been waited for by a thread of the CTA
that receives it: an arrival that is still on its way when that CTA leaves lands in whatever runs there next.  The roles of
both CTAs are played to their ends for every arrangement of short cases: no wait may be left hanging, and no phase of
any barrier may be left that nobody of its CTA has seen.  With every stage's release and every accumulator's drain
announced, also those that nothing follows, some are."""
import itertools

import pytest

LEADER, PEER = 0, 1


class Barriers:
    def __init__(self, count):
        self.count, self.arrived, self.seen = count, {}, {}

    def arrive(self, bar, n=1):
        self.arrived[bar] = self.arrived.get(bar, 0) + n

    def phases(self, bar, extra):
        """Completed phases; `extra` = bytes (in loads) that each phase expects besides its arrivals."""
        left, done = self.arrived.get(bar, 0), 0
        while True:
            need = self.count[bar[1]] + (extra[done] if done < len(extra) else 0)
            if left < need:
                return done, left
            left, done = left - need, done + 1


def play(tiles, KB, S, G, always):
    """`tiles`: accumulators (1 or 2) of each tile of the pair.  Returns the barriers with phases or arrivals unseen."""
    b = Barriers({"full": 8 + 1, "free": 1, "acc_full": 1, "acc_empty": 16})
    n_it = len(tiles) * KB
    loads = {}   # of each use of a stage's slot: activation tiles of both CTAs
    for it in range(n_it):
        loads.setdefault(("full", it % S), []).append(2 * tiles[it // KB])

    def activations(cta):
        for it in range(n_it):
            if it >= S:
                yield (cta, "free", it % S), it // S - 1
            b.arrive((LEADER, "full", it % S), (1 if cta == LEADER else 0) + tiles[it // KB])

    def expansion(cta, g):
        for it in range(g, n_it, G):
            if it >= S:
                yield (cta, "free", it % S), it // S - 1
            b.arrive((LEADER, "full", it % S), 4)

    def commit(name, i):
        for cta in (LEADER, PEER):
            b.arrive((cta, name, i))

    def issuer():
        it = used1 = 0
        for j, halves in enumerate(tiles):
            if j >= 1:
                yield (LEADER, "acc_empty", 0), j - 1
            if halves == 1:
                for _ in range(KB):
                    yield (LEADER, "full", it % S), it // S
                    if always or it + S < n_it:
                        commit("free", it % S)
                    it += 1
                commit("acc_full", 0)
                continue
            free1, i, skew = used1 == 0, 0, S - 1
            while i < KB:
                d = 1
                if i == 0 and not free1:
                    d = min(KB, skew)
                elif KB - i <= skew:
                    d = KB - i
                last = i + d == KB
                for k in range(d):
                    yield (LEADER, "full", (it + k) % S), (it + k) // S
                if last:
                    commit("acc_full", 0)
                if not free1:
                    yield (LEADER, "acc_empty", 1), used1 - 1
                    free1 = True
                for k in range(d):
                    if always or it + k + S < n_it:
                        commit("free", (it + k) % S)
                if last:
                    commit("acc_full", 1)
                it, i = it + d, i + d
            used1 += 1

    def epilogue(cta):
        used1 = 0
        for j, halves in enumerate(tiles):
            for h in range(halves):
                yield (cta, "acc_full", h), (j if h == 0 else used1)
                used1 += h
                if always or j < (len(tiles) - 1 if h == 0 else max(i for i, n in enumerate(tiles) if n == 2)):
                    b.arrive((LEADER, "acc_empty", h))

    threads = [issuer()]
    for cta in (LEADER, PEER):
        threads += [activations(cta)] + [expansion(cta, g) for g in range(G)] + [epilogue(cta) for _ in range(8)]
    waits = [next(t, None) for t in threads]
    moved = True
    while moved:
        moved = False
        for k, t in enumerate(threads):
            while waits[k] is not None:
                bar, phase = waits[k]
                done, _ = b.phases(bar, loads.get(bar[1:], []))
                if done <= phase:
                    break
                assert done == phase + 1, "a wait that tells phases apart by parity passes on the wrong one"
                b.seen[bar] = max(b.seen.get(bar, 0), phase + 1)
                waits[k] = next(t, None)
                moved = True
    assert all(w is None for w in waits), "a wait that nothing ends"
    out = set()
    for bar in b.arrived:
        done, left = b.phases(bar, loads.get(bar[1:], []))
        if left or done > b.seen.get(bar, 0):
            out.add(bar[:2])
    return out


CASES = [(KB, S, G, halves) for KB in (1, 2, 3, 4, 5, 9) for (S, G, halves) in ((6, 3, (1,)), (4, 4, (1, 2)))]


@pytest.mark.parametrize("KB,S,G,halves", CASES)
def test_nothing_is_on_its_way_when_a_cta_leaves(KB, S, G, halves):
    for n in range(0, 5):
        for tiles in itertools.product(halves, repeat=n):
            assert play(tiles, KB, S, G, always=False) == set(), tiles


@pytest.mark.parametrize("KB,S,G,halves", CASES)
def test_announced_without_need_something_is(KB, S, G, halves):
    for tiles in itertools.product(halves, repeat=2):
        assert play(tiles, KB, S, G, always=True) >= {(LEADER, "acc_empty"), (LEADER, "free"), (PEER, "free")}
