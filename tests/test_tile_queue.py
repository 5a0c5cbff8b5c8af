"""The expert launch's tile queue: a model of its hand-back barriers (one mbarrier
per slot, on which every reader of an entry arrives) under random schedules in
which the readers fall behind one another as far as the barriers let them.  The
gather warps leave the queue at the first tile that is not gathered; a slot must
be filled again only after every remaining reader has read it."""
import random
import re
from pathlib import Path

import pytest

SRC = (Path(__file__).resolve().parent.parent / "paper_2608_06690_gb300/csrc/k_experts_tc.cu").read_text()
SLOTS = int(re.search(r"constexpr int kTQ = (\d+);", SRC).group(1))
GROUPS = int(re.search(r"constexpr int kGatherGroups = (\d+);", SRC).group(1))
# readers of an entry: per CTA the weight warp, four epilogue warps and the
# gather warps; the leader's MMA warp and the other CTA's token warp
GATHER = {"cp_async": 2 * 4 * GROUPS, "gather4": 2}
OTHERS = 2 * (2 + 4)


class Barrier:
    def __init__(self, count):
        self.phase, self.expected, self.pending = 0, count, count

    def arrive(self, drop=False):
        self.expected -= drop
        self.pending -= 1
        if self.pending == 0:
            self.phase += 1
            self.pending = self.expected

    def passed(self, parity):
        return self.phase & 1 != parity


class Overwritten(Exception):
    pass


def run(entries, gathered, n_gather, leave, rng):
    """entries tiles, the first `gathered` of them gathered, then the list's end."""
    bars = [Barrier(OTHERS + n_gather) for _ in range(SLOTS)]
    pushed = 0
    at = [0] * (OTHERS + n_gather)      # the next entry of each reader (the first n_gather gather rows)
    done = [False] * len(at)
    slow = rng.sample(range(len(at)), len(at) // 2)

    def step(r):
        """Reader r reads its next entry, if it is published; False if it cannot."""
        nonlocal pushed
        e = at[r]
        if done[r] or e >= pushed:
            return False
        if pushed - 1 - e >= SLOTS:
            raise Overwritten(f"reader {r}: entry {e} replaced by {e + SLOTS}")
        end = e == entries
        at[r] += 1
        if r < n_gather and e >= gathered:
            done[r] = leave(bars, e, end, e - gathered)
        else:
            bars[e % SLOTS].arrive()
            done[r] = end
        return True

    def push():
        nonlocal pushed
        if pushed > entries or not bars[pushed % SLOTS].passed((pushed // SLOTS & 1) ^ 1):
            return False
        pushed += 1
        return True

    while not all(done):
        readers = list(range(len(at)))
        rng.shuffle(readers)
        if rng.random() < 0.9:  # the slow ones rarely come first
            readers.sort(key=lambda r: r in slow)
        # the leader goes as far as it may before a reader moves, most of the time
        moved = push() if rng.random() < 0.7 else False
        if not moved and not any(step(r) for r in readers) and not push():
            raise Overwritten("the leader waits for a phase that no reader completes")
    return bars


def drop_slot_by_slot(bars, e, end, k):
    bars[e % SLOTS].arrive(drop=True)
    return end or k == SLOTS - 1


def drop_all_at_once(bars, e, end, k):
    for b in bars:
        b.arrive(drop=True)
    return True


@pytest.mark.parametrize("form", list(GATHER))
@pytest.mark.parametrize("gathered", [0, 1, 3, SLOTS, 21])
@pytest.mark.parametrize("more", [0, 1, SLOTS - 1, SLOTS, 40])
def test_slot_refilled_only_after_every_reader(form, gathered, more):
    for seed in range(8):
        bars = run(gathered + more, gathered, GATHER[form], drop_slot_by_slot, random.Random(seed))
        assert all(b.pending > 0 for b in bars)
        assert more + 1 < SLOTS or all(b.expected == OTHERS for b in bars)


def test_the_model_shows_a_second_arrival():
    """Leaving every slot at the first other tile, the warps arrive a second time
    on slots that slower readers have yet to read, and the slots come back early."""
    hits = 0
    for seed in range(20):
        try:
            run(43, 3, GATHER["cp_async"], drop_all_at_once, random.Random(seed))
        except Overwritten:
            hits += 1
    assert hits


def test_leaving_warps_drop_the_published_slot():
    """The kernel's only drop names the slot of the entry that it has waited for."""
    drops = re.findall(r"mbar_arrive_drop\(dsmem_addr\(tq_empty_bar\((.+?)\), 0\)\)", SRC)
    assert drops == ["e % kTQ"]
