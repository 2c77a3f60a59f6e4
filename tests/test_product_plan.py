"""How the product kernel's launches are laid out, from the code that lays them out (host functions of the kernel's header,
compiled into a small program that runs on the CPU)."""
import os
import subprocess

import pytest

from paper_2510_07535_b200 import build as owl_build

FIELDS = ("rounds", "tall_rounds", "h_lo", "group_rows", "stages", "kblocks_per_stage", "smem", "rows_on_lanes_argmax",
          "rows_on_lanes_store")
PROGRAM = r"""
#include <cstdio>
#include "gemm_umma.cuh"
int main() {
    using namespace owl::gemm_path;
    int M, N, K, sms;
    while (scanf("%d %d %d %d", &M, &N, &K, &sms) == 4) {
        const int groups = column_groups(M);
        const GemmParams g = product_plan(M, N, K, product_pairs(N, sms));
        printf("%d %d %d %d %d %d %d %d %d\n", g.rounds, g.tall_rounds, g.h_lo, g.group_rows, g.stages, stage_kblocks(groups),
               smem_bytes(groups, g.stages, g.block_bytes), rows_on_lanes(g, kEpiArgmax), rows_on_lanes(g, kEpiStore));
    }
}
"""


@pytest.fixture(scope="session")
def plans(tmp_path_factory):
    """Maps [(M, N, K), ...] to their plans on 148 SMs."""
    where = tmp_path_factory.mktemp("plan")
    source, program = where / "plan.cu", where / "plan"
    source.write_text(PROGRAM)
    subprocess.check_call([owl_build.NVCC, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static",
                           f"-I{owl_build.CSRC}", "-o", str(program), str(source)], env={**os.environ, "TMPDIR": str(where)})

    def of(shapes):
        asked = "".join(f"{m} {n} {k} 148\n" for m, n, k in shapes)
        out = subprocess.run([str(program)], input=asked, capture_output=True, text=True, check=True).stdout
        return [dict(zip(FIELDS, map(int, line.split()))) for line in out.splitlines()]
    return of


def test_an_sm_never_holds_two_ctas(plans):
    """Each takes all of its SM's tensor memory, a pair that of two SMs: two pairs that share two SMs could each hold one
    half and wait for the other.  228 KB per SM, 1 KB of each CTA's reserved."""
    shapes = [(m, n, 4096) for m in range(1, 385) for n in (1, 16, 512, 1184, 2048, 4096, 5076, 8192, 16384, 49152, 128256)]
    for shape, p in zip(shapes, plans(shapes)):
        assert 2 * (p["smem"] + 1024) > 228 * 1024 and p["smem"] <= 227 * 1024, (shape, p)
        assert p["stages"] >= 2 and p["h_lo"] + (16 if p["tall_rounds"] else 0) <= 256, (shape, p)


# (rows of A, K, d) of cell calls: products of 4d weight rows that test_gpu_kernel_edges.py checks element by element
SEVERAL_TILES = [(10, 1088, 12288 + 252), (130, 1088, 12288 + 252), (200, 1088, 12288 + 252), (257, 1088, 12288 + 252), (384, 1024, 12288 + 252)]
ROWS_ON_LANES = [(64, 1088, 1184), (100, 448, 1184), (256, 1088, 1184), (256, 1088, 12288 + 252), (257, 1088, 1184), (384, 1024, 1184),
                 (384, 960, 2048), (33, 64, 4)]


def test_the_shapes_of_the_gpu_tests_have_what_they_are_there_for(plans):
    """Three rounds of tiles and more, the last ones lower, a ring that wraps within a tile, an odd number of k-blocks; and the
    swapped operand order at one and at two groups, at one round and at several."""
    for (m, k, d), p in zip(SEVERAL_TILES, plans([(m, 4 * d, k) for m, k, d in SEVERAL_TILES])):
        assert p["rounds"] >= 3 and 0 < p["tall_rounds"] < p["rounds"], p
        assert -(-(k // 64) // p["kblocks_per_stage"]) > p["stages"], p
        assert not p["rows_on_lanes_store"], p
    assert any((k // 64) % 2 for _, k, _ in SEVERAL_TILES) and {m > 256 for m, _, _ in SEVERAL_TILES} == {True, False}
    lanes = plans([(m, 4 * d, k) for m, k, d in ROWS_ON_LANES])
    assert all(p["rows_on_lanes_store"] for p in lanes)
    assert {(p["kblocks_per_stage"], p["rounds"] > 1) for p in lanes} >= {(2, False), (2, True), (1, False)}
