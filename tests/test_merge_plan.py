"""Which blocks of rows the merge kernel's CTAs take where they go by the places at which the line of key tiles is cut, from the
code that decides it (host side of the kernel's headers, compiled into a small program that runs on the CPU)."""
import os
import random
import subprocess

import pytest

from paper_2510_07535_b200 import build as owl_build

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "combine.cuh"
using namespace owl;
int main() {
    int B, H, ctas, turns;
    while (scanf("%d %d %d %d", &B, &H, &ctas, &turns) == 4) {
        std::vector<int> tiles(B);
        long long sum = 0;
        int units = 0, lo = 1 << 30, hi = 0;
        for (int& t : tiles) {
            scanf("%d", &t);
            if (t) { sum += (long long)t * H; units += H; lo = t < lo ? t : lo; hi = t > hi ? t : hi; }
        }
        const int uniform = units && lo == hi ? lo : 0;
        Partition<long long> part;
        part.init(sum, ctas, units, uniform);
        Partition<int> small;
        small.init((int)sum, ctas, units, uniform);
        std::vector<long long> begin(B + 1, 0);
        for (int b = 0; b < B; ++b) begin[b + 1] = begin[b] + (tiles[b] ? (long long)(tiles[b] + part.pen) * H : 0);
        int differ = begin[B] != part.total || small.total != (int)part.total || small.pen != part.pen;
        for (int c = 0; c < ctas; ++c) {
            long long t0, t1; int s0, s1;
            part.range(c, t0, t1); small.range(c, s0, s1);
            differ += s0 != t0 || s1 != t1;
            printf("%lld %lld ", t0, t1);
        }
        for (long long t = 0; t < part.total; ++t) differ += part.owner(t) != small.owner((int)t);
        printf("\n%d %d\n", part.pen, differ);
        for (int i = 0; i < combine_cuts(ctas) * turns; ++i) {
            const int turn = i / combine_cuts(ctas), cut = i % combine_cuts(ctas) + 1;
            long long t, t_end;
            part.range(cut, t, t_end);
            int b = 0, h, len, first, stride;
            if (t >= part.total) continue;
            while (begin[b + 1] <= t) ++b;
            if (!cut_unit(part, t, begin[b], begin[b + 1], H, h, len)) continue;
            const long long first_tile = begin[b] + (long long)h * len + part.pen;
            const int c0 = part.owner(first_tile), c1 = part.owner(first_tile + tiles[b] - 1);
            cut_share(cut, c0, c1 - c0 + 1, turn, turns, first, stride);
            printf("%d %d %d %d ", b, h, first, stride);
        }
        printf("\n");
    }
}
"""


@pytest.fixture(scope="session")
def program(tmp_path_factory):
    where = tmp_path_factory.mktemp("merge_plan")
    source, path = where / "plan.cu", where / "plan"
    source.write_text(PROGRAM)
    subprocess.check_call([owl_build.NVCC, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static",
                           f"-I{owl_build.CSRC}", "-o", str(path), str(source)], env={**os.environ, "TMPDIR": str(where)})
    return str(path)


def test_every_block_of_every_unit_that_is_cut_is_taken_once(program):
    """Units that lie in several pieces, found by going through the pieces tile by tile: each of their blocks has one CTA, no
    other unit has any, and the 32-bit schedule cuts like the 64-bit one."""
    rng = random.Random(7)
    cases = []
    for _ in range(400):
        batch, heads = rng.choice([1, 2, 3, 31, 33, 64, 100]), rng.choice([1, 2, 8])
        most = rng.choice([1, 2, 5, 40, 300])
        tiles = [rng.randint(1, most) for _ in range(batch)]
        if rng.random() < 0.3:
            tiles = [tiles[0]] * batch                                   # the cut that follows the units' boundaries
        elif rng.random() < 0.4:
            tiles = [0 if rng.random() < 0.2 else t for t in tiles]      # refused sequences
        cases.append((batch, heads, rng.choice([148, 148, 148, 132, 16, 2, 1]), rng.randint(1, 4), tiles))
    asked = "".join(f"{b} {h} {c} {t} {' '.join(map(str, tiles))}\n" for b, h, c, t, tiles in cases)
    lines = subprocess.run([program], input=asked, capture_output=True, text=True, check=True).stdout.split("\n")
    cut_units = aligned = 0
    for (batch, heads, ctas, _, tiles), ranges, checks, taken in zip(cases, lines[0::3], lines[1::3], lines[2::3]):
        edges = list(map(int, ranges.split()))
        assert edges[2::2] == edges[1:-1:2]                              # one piece ends where the next begins
        pen, differ = map(int, checks.split())
        assert differ == 0
        aligned += pen == 0
        starts, blocks = set(edges[2::2]), 5                             # of eight rows, in every unit
        want, at = {}, 0
        for b in range(batch):
            for h in range(heads if tiles[b] else 0):
                first = at + pen
                if any(first < place < first + tiles[b] for place in starts):
                    want.update({(b, h, k): 1 for k in range(blocks)})
                    cut_units += 1
                at = first + tiles[b]
        got, words = {}, list(map(int, taken.split()))
        for b, h, first, stride in zip(*[iter(words)] * 4):
            for k in range(first, blocks, stride):
                got[b, h, k] = got.get((b, h, k), 0) + 1
        assert got == want
    assert cut_units > 1000 and aligned > 10
