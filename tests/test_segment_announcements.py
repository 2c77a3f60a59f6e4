"""A model of how the attention kernel's roles agree on the segments of a CTA's piece and hand over P tile by tile, run under
random interleavings on the CPU.  A wait on a tile or on a free slot may give up at any point; from then on all of those
return at once.  What is never abortable must still end: the hardware barriers, the wait for a score tile and the producer's
look at `seg_reached`; every reader must have taken every segment; a copy goes to the ring slot of its own tile and kind; and
nobody writes over the scores of a segment whose products are under way."""
import random
import re
from pathlib import Path

import pytest

SOURCE = (Path(__file__).parent.parent / "paper_2510_07535_b200" / "csrc" / "verify_attn_umma.cuh").read_text()
PLACES = int(re.search(r"constexpr int kSegs = (\d+);", SOURCE).group(1))
SLOTS = int(re.search(r"constexpr int kSlots = (\d+);", SOURCE).group(1))
SLOTS_NARROW = int(re.search(r"constexpr int kSlotsNarrow = (\d+);", SOURCE).group(1))
# the condition under which a warp writes its maximum and sums over its scores at a segment's end
EXCHANGE = re.search(r"if \((.*)\) \{\s*const uint32_t mine\[4\]", SOURCE).group(1)


class Cta:
    def __init__(self, rng, segments, paced, certain, by_tile, idle_aside="!idle" in EXCHANGE, slots=SLOTS):
        self.idle_aside, self.slots = idle_aside, slots
        self.rng, self.paced, self.certain, self.by_tile, self.abort = rng, paced, certain, by_tile, False
        self.tiles = [rng.randint(1, 3) for _ in range(segments)] + [0]       # 0: no more segments
        self.place, self.announced = [None] * PLACES, [0] * PLACES            # contents; completed phases
        self.reached = 0
        self.copied, self.freed = set(), 0                                    # items (K, V, K, V, ...) copied; tiles consumed
        self.q_full = 0                                                       # segments whose Q has been loaded
        self.live = [rng.randint(1, 4) for _ in range(segments + 1)]          # softmax warps that hand over P
        self.scores = self.products = 0                                       # tiles: S announced, P V done
        self.open, self.generation = {}, {1: 0, 3: 0, 4: 0}                   # hardware barriers: (arrived, expected)

    def arrive(self, bar, warps, need):          # bar.arrive
        got, expected = self.open.pop(bar, (0, need))
        got += warps
        assert expected == need and got <= need, f"barrier {bar}: {got} of {need} and {expected} warps in one generation"
        if got == need:
            self.generation[bar] += 1
        else:
            self.open[bar] = (got, need)

    def sync(self, bar, need):                   # bar.sync of one warp (of one role for barriers 1 and 3)
        mine = self.generation[bar]
        self.arrive(bar, 1, need)
        return lambda: self.generation[bar] > mine

    def bounded(self, condition):
        return lambda: condition() or self.abort

    def complete(self, k):                       # try_wait.parity on the announcement barrier
        return lambda: self.announced[k % PLACES] % 2 != (k // PLACES) % 2

    def producer(self):
        item, wanted = 0, 0                      # the ring's count; of the sequence K, V, K, V, ...
        for k, tiles in enumerate(self.tiles):
            if self.paced and k >= PLACES:
                yield lambda: self.reached >= k - PLACES + 1
            self.place[k % PLACES] = k
            yield None
            self.announced[k % PLACES] += 1
            for _ in range(2 * tiles):
                free = lambda: item - 2 * self.freed < self.slots
                yield self.bounded(free)
                if free():
                    assert item % 2 == wanted % 2, "K in a slot of V"
                    self.copied.add(item)
                if free() or self.by_tile:
                    item += 1
                wanted += 1

    def meet(self, k, leader):                   # meet_before_segment
        if self.paced:
            if leader:
                yield self.complete(k)
            yield self.sync(3, 4)
        else:
            yield self.complete(k)               # every reader for itself
        yield None

    def mma(self, taken):
        for k in range(len(self.tiles)):
            yield from self.meet(k, False)
            taken.append(self.place[k % PLACES])
            yield self.bounded(lambda: self.q_full > k)
            for _ in range(self.tiles[taken[-1]]):
                first = self.products
                yield self.bounded(lambda: {2 * first, 2 * first + 1} <= self.copied)
                self.scores += 1
                yield self.sync(4, self.live[taken[-1]] + 1)
                self.products += 1
                self.freed = self.products

    def softmax(self, taken, leader):
        """One stream's warpgroup; the second one here only loads Q and sleeps through the tiles."""
        yield from self.meet(0, leader)
        for k in range(len(self.tiles)):
            seg = self.place[k % PLACES]
            taken.append(seg)
            if self.tiles[seg] == 0:
                return
            yield self.sync(1, 3)                # the Q blocks are free
            if leader:
                self.reached = k
            yield self.sync(1, 3)                # the tree's masks
            if leader:
                self.q_full += 1
                base = sum(self.tiles[:seg])
                for i in range(self.tiles[seg]):
                    announced = lambda: self.scores > base + i
                    yield announced if self.certain else self.bounded(announced)
                    self.arrive(4, self.live[seg], self.live[seg] + 1)
                finished = lambda: self.products >= base + self.tiles[seg]
                yield finished if self.certain else self.bounded(finished)
            yield from self.meet(k + 1, leader)
            assert not self.paced or self.place[k % PLACES] == seg        # bad_page is read here

    def idle(self):
        """The softmax warps without a row of the unit, if there are any: from the masks straight to the segment's end."""
        yield from self.meet(0, False)
        for k in range(len(self.tiles)):
            seg = self.place[k % PLACES]
            if self.tiles[seg] == 0:
                return
            yield self.sync(1, 3)
            yield self.sync(1, 3)
            if self.live[seg] < 4 and not self.idle_aside:
                assert self.abort or self.products >= sum(self.tiles[:seg + 1]), "scores overwritten under the products"
            yield from self.meet(k + 1, False)

    def run(self, abort_at):
        taken = [[], [], []]
        roles = {r: next(r) for r in (self.producer(), self.mma(taken[0]), self.softmax(taken[1], True), self.softmax(taken[2], False),
                                      self.idle())}
        step = 0
        while roles:
            self.abort = self.abort or step >= abort_at
            ready = [r for r, wait in roles.items() if wait is None or wait()]
            if not ready:
                assert not self.abort, "hang"
                abort_at = step                  # nothing moves any more: the first wait gives up
                continue
            step += 1
            r = ready[0] if self.rng.random() < 0.6 else self.rng.choice(ready)      # runs of one role, and mixtures
            try:
                roles[r] = next(r)
            except StopIteration:
                del roles[r]
        return taken


def segments_of(seed, segments, paced=True, certain=True, by_tile=True, **more):
    rng = random.Random(seed)
    return Cta(rng, segments, paced, certain, by_tile, **more).run(abort_at=rng.choice([0, 10 ** 9, rng.randint(0, 12 * segments)]))


@pytest.mark.parametrize("segments", [1, PLACES - 1, PLACES, PLACES + 1, 16, 40])
def test_all_roles_take_the_same_segments_whatever_gives_up(segments):
    for seed in range(300):
        assert segments_of(seed, segments) == [list(range(segments + 1))] * 3, seed


@pytest.mark.parametrize("segments", [1, PLACES + 1, 40])
def test_the_same_with_the_longer_ring_of_narrow_units(segments):
    for seed in range(300):
        assert segments_of(seed, segments, slots=SLOTS_NARROW) == [list(range(segments + 1))] * 3, seed


@pytest.mark.parametrize("segments,without", [(40, "paced"), (4, "certain"), (4, "by_tile"), (4, "idle_aside")])
def test_the_model_shows_what_each_rule_is_for(segments, without):
    """A producer that nothing paces, softmax warps that hand over P of a tile whose S was not announced, a producer that
    counts only what it has copied, idle warps that take part in the exchange at a segment's end."""
    def broken(seed):
        try:
            return segments_of(seed, segments, **{without: False}) != [list(range(segments + 1))] * 3
        except (AssertionError, IndexError):
            return True
    assert any(broken(seed) for seed in range(300))
