"""The order of a resident launch's blocks, on the host.

A model of how the workers and the tail of the resident kernel
(csrc/step_resident.cu) wait for one another: a worker reports its arrival at a
step with its candidates, writes its sums when the tail has taken those of
kResRows steps before, waits for all arrivals, and for the tail when the step
has candidates.  The tail waits for all arrivals, finishes the candidates, then
takes the step's sums.  The number of rows and of arrival words come from the
sources.  Whatever the speed of each block, every block must count exactly the
candidates of the step, and none may wait for ever.
"""
import os
import random
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0704_0043_gb300", "csrc",
                   "internal.h")


def constant(name, default=None):
    with open(SRC) as f:
        m = re.search(r"constexpr int %s = (\d+);" % name, f.read())
    return int(m.group(1)) if m else default


class Launch:
    def __init__(self, workers, cands):
        self.W, self.cands = workers, cands  # cands[s][w]
        self.rows, self.slots = constant("kResRows"), constant("kResSlots", 1)
        self.count, self.total = [0] * self.slots, [0] * self.slots
        self.rows_in = [0] * self.rows
        self.done = self.stats_done = 0

    def arrivals(self, s, seen):
        slot = s % self.slots
        while self.count[slot] < self.W * (s // self.slots + 1):
            yield
        n = self.total[slot] - seen[slot]
        seen[slot] = self.total[slot]
        assert n == sum(self.cands[s]), "step %d counts the candidates of another" % s
        return n

    def worker(self, w):
        seen = [0] * self.slots
        for s in range(len(self.cands)):
            yield
            self.count[s % self.slots] += 1
            self.total[s % self.slots] += self.cands[s][w]
            yield
            while s >= self.rows and self.stats_done < s - self.rows + 1:
                yield
            self.rows_in[s % self.rows] += 1
            n = yield from self.arrivals(s, seen)
            while n > 0 and self.done < s + 1:
                yield

    def tail(self):
        seen = [0] * self.slots
        for s in range(len(self.cands)):
            yield
            if (yield from self.arrivals(s, seen)) > 0:
                yield
                self.done = s + 1
            while self.rows_in[s % self.rows] < self.W * (s // self.rows + 1):
                yield
            yield
            self.stats_done = s + 1


@pytest.mark.parametrize("seed", range(40))
def test_every_block_counts_the_steps_own_candidates(seed):
    r = random.Random(seed)
    workers, steps = r.randrange(1, 6), 60
    cands = [[r.randrange(1, 4) if r.random() < 0.3 else 0 for _ in range(workers)] if r.random() < 0.4
             else [0] * workers for _ in range(steps)]
    launch = Launch(workers, cands)
    blocks = [launch.worker(w) for w in range(workers)] + [launch.tail()]
    turns = 0
    while blocks:
        # one block is held up for a while, as far as the others come without it
        late = r.choice(blocks)
        for _ in range(r.randrange(1, 400)):
            b = late if len(blocks) == 1 or r.random() < 0.002 else r.choice([x for x in blocks if x is not late])
            try:
                next(b)
            except StopIteration:
                blocks.remove(b)
                break
        turns += 1
        assert turns < 4000, "blocks wait for one another"
