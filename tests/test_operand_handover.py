"""Hand-over of the tensor-core kernel's i-side operand buffers, on the CPU.

The loader fills two buffers in turn; whoever waits for a fill does so by the
parity of its barrier, so nobody may be lapped by two fills.  The barriers of
the hand-over are played through with one warp starved: it takes a step only
when no other warp can.  How many arrivals empty a buffer, and which roles make
them, is read from the kernel's source.  Items of one tile, in which only the
first group of warps has work: an issuer of another group does nothing but wait
and arrive.
"""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1204_6630_gb300", "csrc", "count_tc.cu")
WORK, GROUPS, ITEMS = 16, 4, 24


class Barrier:
    def __init__(self, count):
        self.count = self.pending = count
        self.phase = 0

    def arrive(self):
        self.pending -= 1
        assert self.pending >= 0
        if self.pending == 0:
            self.pending = self.count
            self.phase += 1

    def done(self, parity):  # as the parity forms of the wait: true when that phase is the one before the current
        return (self.phase & 1) != parity


def protocol():
    """(arrivals that empty a buffer, whether the classifying warps make one, whether the issuers do)."""
    src = open(SRC).read()
    count = re.search(r"mbar_init\(a_empty \+ k, ([^)]*)\)", src).group(1)
    names = {"kWorkWarps": str(WORK), "kGroups": str(GROUPS)}
    count = sum(int(names[t.strip()]) for t in count.split("+"))
    work, issue = (re.search(r"=+ %s\n(.*?)// =+ %s" % ends, src, re.S).group(1)
                   for ends in (("classifying warps", "mma issuers"), ("mma issuers", "loader")))
    return count, "mbar_arrive(a_empty" in work, "mbar_arrive(a_empty" in issue


@pytest.mark.parametrize("starved", ["worker 0", "worker 7", "issuer 0", "issuer 2", "loader"])
@pytest.mark.parametrize("stages", [4, 6, 8])
def test_no_warp_can_be_lapped(stages, starved):
    count, workers_arrive, issuers_arrive = protocol()
    a_full, a_empty = [Barrier(1), Barrier(1)], [Barrier(count), Barrier(count)]
    full, empty = ([Barrier(c) for _ in range(stages)] for c in (1, WORK + GROUPS))
    d_full, d_free = Barrier(1), Barrier(WORK // GROUPS)

    def loader():
        for k in range(ITEMS):
            yield a_empty[k & 1], ((k >> 1) & 1) ^ 1
            a_full[k & 1].arrive()
            yield empty[k % stages], ((k // stages) & 1) ^ 1
            full[k % stages].arrive()

    def issuer(g):
        for k in range(ITEMS):
            yield full[k % stages], (k // stages) & 1
            yield a_full[k & 1], (k >> 1) & 1
            if g == 0:
                yield d_free, (k & 1) ^ 1
                d_full.arrive()
            if issuers_arrive:
                a_empty[k & 1].arrive()
            empty[k % stages].arrive()

    def worker(w):
        for k in range(ITEMS):
            yield full[k % stages], (k // stages) & 1
            if w < WORK // GROUPS:
                yield d_full, k & 1
                d_free.arrive()
            if workers_arrive:
                a_empty[k & 1].arrive()
            empty[k % stages].arrive()

    roles = {"loader": loader(), **{f"issuer {g}": issuer(g) for g in range(GROUPS)},
             **{f"worker {w}": worker(w) for w in range(WORK)}}
    waits = {n: next(r) for n, r in roles.items()}
    while waits:
        ready = [n for n, (bar, parity) in waits.items() if bar.done(parity)]
        assert ready, f"nobody can go on: {sorted(waits)}"
        n = next((n for n in ready if n != starved), ready[0])
        try:
            waits[n] = next(roles[n])
        except StopIteration:
            del waits[n]
