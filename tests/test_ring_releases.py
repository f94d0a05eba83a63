"""A randomised model of the binary64 kernel's ring in a cluster (no GPU).

Every stage of a CTA (cy, cx) of a cm x cn cluster is filled by multicast: one piece of
A from column 0 of its row, and the pieces of B of its column, piece j from row
j mod cm.  A CTA issues its copies into a stage, and expects its own bytes there, when
the stage's "empty" barrier says that the last contents were released; a warp that has
read a stage arrives on the empty barriers of the CTAs that filled it, and on its own.
A barrier counts arrivals whoever they come from.  The kernel counts those of the whole
cluster row and column (`everyone`), more than the copies reach; the exact count is the
CTA itself, its row mates where it sends A, its column mates where it sends B.  Copies
and arrivals take any time here.  Checked: nothing lands in a stage that is still being
read, no barrier gets an arrival too many, the waits' parities tell the phases apart,
and nothing deadlocks.  The kernel's counts hold where every row sends a piece of B, or
with one column; else a CTA that waits for nobody in a row without pieces arrives a
second time in the place of one that has not released yet."""
import random

import pytest


class Barrier:
    def __init__(self, count):
        self.count = self.pending = count
        self.done = 0           # completed phases
        self.tx = 0             # bytes still to come (pieces); below 0 before expect_tx

    def arrive(self, tx=0):
        assert self.pending > 0, "an arrival too many in a phase"
        self.pending -= 1
        self.tx += tx
        self.settle()

    def land(self):
        self.tx -= 1
        self.settle()

    def settle(self):
        if self.pending == 0 and self.tx == 0:
            self.done += 1
            self.pending = self.count


def wait(bar, phase):
    """Whether a wait for completed phase `phase` (from 0) passes, by parity."""
    assert phase <= bar.done <= phase + 1, "the parity is ambiguous"
    return bar.done == phase + 1


def run(cm, cn, pieces, stages, steps, warps, seed, everyone):
    rnd = random.Random(seed)
    ctas = [(y, x) for y in range(cm) for x in range(cn)]
    row = {c: [(c[0], x) for x in range(cn)] for c in ctas}
    col = {c: [(y, c[1]) for y in range(cm)] for c in ctas}
    sends_a = {c: c[1] == 0 for c in ctas}
    sends_b = {c: len(range(c[0], pieces, cm)) for c in ctas}
    reach = {c: {c} | set(row[c] if everyone or sends_a[c] else ())
             | set(col[c] if everyone or sends_b[c] else ()) for c in ctas}
    fills = {c: [s for s in ctas if c in reach[s]] for c in ctas}
    full = {c: [Barrier(1) for _ in range(stages)] for c in ctas}
    empty = {c: [Barrier(warps * len(reach[c])) for _ in range(stages)] for c in ctas}
    issued = {c: 0 for c in ctas}
    read = {(c, w): 0 for c in ctas for w in range(warps)}     # steps released
    reading = {k: False for k in read}
    slow = {k: rnd.choice((1, 1, 1, 12)) for k in read}        # some warps fall behind
    flight = []
    idle = 0
    while min(read.values()) < steps or flight:
        idle += 1
        assert idle < 20000, "deadlock"
        kind = rnd.randrange(3)
        if kind == 0 and flight:
            flight.pop(rnd.randrange(len(flight)))()
            idle = 0
        elif kind == 1:
            c = rnd.choice(ctas)
            n = issued[c]
            if n == steps or not (n < stages or wait(empty[c][n % stages], n // stages - 1)):
                continue
            full[c][n % stages].arrive(1 + pieces)
            for d, count in [(d, 1) for d in row[c] if sends_a[c]] + [(d, sends_b[c]) for d in col[c]]:
                def land(d=d, n=n):
                    assert n < stages or all(read[d, w] > n - stages for w in range(warps)), \
                        "a copy into a stage that is still read"
                    full[d][n % stages].land()
                flight += [land] * count
            issued[c] += 1
            idle = 0
        elif kind == 2:
            k = rnd.choice(list(read))
            if rnd.randrange(slow[k]) or read[k] == steps:
                continue
            c, n = k[0], read[k]
            if not reading[k]:
                reading[k] = wait(full[c][n % stages], n // stages)
                continue
            reading[k] = False
            read[k] += 1
            flight += [lambda b=empty[s][n % stages]: b.arrive() for s in fills[c]]
            idle = 0


CLUSTERS = [(1, 1), (1, 2), (2, 1), (2, 2), (4, 1), (1, 4), (3, 2), (4, 4), (2, 8), (8, 2), (5, 3),
            (6, 2), (16, 1), (1, 16)]


# pieces: 8 of strips of 128 columns, 4 of strips of 64
@pytest.mark.parametrize("cm,cn,pieces,everyone", [
    (cm, cn, pieces, everyone) for cm, cn in CLUSTERS for pieces in (8, 4)
    for everyone in (True, False) if not everyone or cm <= pieces or cn == 1])
def test_releases(cm, cn, pieces, everyone):
    for seed in range(24):
        run(cm, cn, pieces, (2, 4)[seed % 2], 9, (1, 2)[seed // 2 % 2], seed, everyone)


@pytest.mark.parametrize("cm,cn", [(8, 2), (5, 3), (6, 2)])
def test_counts_of_the_whole_row_and_column_fail_without_pieces(cm, cn):
    failed = 0
    for seed in range(40):
        try:
            run(cm, cn, 4, 2, 9, 1, seed, everyone=True)
        except AssertionError as e:
            assert "still read" in str(e)
            failed += 1
    assert failed >= 5
