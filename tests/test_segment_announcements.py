"""A model of how the attention kernel's roles agree on the segments of a CTA's piece and hand over P tile by tile, run under
random interleavings on the CPU.  A wait on a tile or on a free slot may give up at any point; from then on all of those
return at once.  What is never abortable must still end: the hardware barriers, the wait for a score tile and the producer's
look at `seg_reached`; every reader must have taken every segment; and the copies that the producer has issued must be
the first ones in order, which is what the drain at the kernel's end takes them for."""
import random
import re
from pathlib import Path

import pytest

SOURCE = (Path(__file__).parent.parent / "paper_2510_07535_b200" / "csrc" / "verify_attn_umma.cuh").read_text()
PLACES = int(re.search(r"constexpr int kSegs = (\d+);", SOURCE).group(1))
SLOTS = int(re.search(r"constexpr int kSlots = (\d+);", SOURCE).group(1))


class Cta:
    def __init__(self, rng, segments, paced, certain, final):
        self.rng, self.paced, self.certain, self.final, self.abort = rng, paced, certain, final, False
        self.tiles = [rng.randint(1, 3) for _ in range(segments)] + [0]       # 0: no more segments
        self.place, self.announced = [None] * PLACES, [0] * PLACES            # contents; completed phases
        self.reached = 0
        self.issued = self.freed = 0                                          # slots copied to; tiles (two slots) consumed
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
        going, slot = True, 0                    # of the sequence K, V, K, V, ...
        for k, tiles in enumerate(self.tiles):
            if self.paced and k >= PLACES:
                yield lambda: self.reached >= k - PLACES + 1
            self.place[k % PLACES] = k
            yield None
            self.announced[k % PLACES] += 1
            for _ in range(2 * tiles):
                free = lambda: self.issued - 2 * self.freed < SLOTS
                if going or not self.final:
                    yield self.bounded(free)
                    going = free()
                if going:
                    assert self.issued == slot, "a copy after one that was left out"
                    self.issued += 1
                slot += 1

    def meet(self, k, leader):                   # meet_before_segment
        if self.paced:
            if leader:
                yield self.complete(k)
            yield self.sync(3, 3)
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
                yield self.bounded(lambda: self.issued >= 2 * first + 2)
                self.scores += 1
                yield self.sync(4, self.live[taken[-1]] + 1)
                self.products += 1
                self.freed = min(self.issued // 2, self.products)

    def softmax(self, taken, leader):
        """One stream's warpgroup; the second one here only loads Q and sleeps through the tiles."""
        yield from self.meet(0, leader)
        for k in range(len(self.tiles)):
            seg = self.place[k % PLACES]
            taken.append(seg)
            if self.tiles[seg] == 0:
                return
            yield self.sync(1, 2)                # the Q blocks are free
            if leader:
                self.reached = k
            yield self.sync(1, 2)                # the tree's masks
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

    def run(self, abort_at):
        taken = [[], [], []]
        roles = {r: next(r) for r in (self.producer(), self.mma(taken[0]), self.softmax(taken[1], True), self.softmax(taken[2], False))}
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


def segments_of(seed, segments, paced=True, certain=True, final=True):
    rng = random.Random(seed)
    return Cta(rng, segments, paced, certain, final).run(abort_at=rng.choice([0, 10 ** 9, rng.randint(0, 12 * segments)]))


@pytest.mark.parametrize("segments", [1, PLACES - 1, PLACES, PLACES + 1, 16, 40])
def test_all_roles_take_the_same_segments_whatever_gives_up(segments):
    for seed in range(300):
        assert segments_of(seed, segments) == [list(range(segments + 1))] * 3, seed


@pytest.mark.parametrize("segments,without", [(40, "paced"), (4, "certain"), (4, "final")])
def test_the_model_shows_what_each_rule_is_for(segments, without):
    """A producer that nothing paces, softmax warps that hand over P of a tile whose S was not announced, a producer that
    copies on after a wait of its own gave up."""
    def broken(seed):
        try:
            return segments_of(seed, segments, **{without: False}) != [list(range(segments + 1))] * 3
        except (AssertionError, IndexError):
            return True
    assert any(broken(seed) for seed in range(300))
