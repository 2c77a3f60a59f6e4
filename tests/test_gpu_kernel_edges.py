"""Kernel branches at the sizes where they can go wrong, against the CPU oracle (tolerances as in test_gpu_parity)."""
import pytest

from paper_2510_07535_b200 import workloads as W
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


def fill_dead_slots(wl):
    """NaN, Inf and huge values in the slots past every sequence's last drafted position (what a cache may hold there)."""
    page = wl.spec.page_size
    for b in range(wl.spec.batch):
        keys = int(wl.ctx_lens[b]) + int(wl.node_offsets[b + 1] - wl.node_offsets[b])
        pg = int(wl.block_table[b, (keys - 1) // page])
        for j in range((keys - 1) % page + 1, page):
            wl.k_cache[pg, :, j, :] = (0x7FC0, 0x7F80, 0xFF80, 0x7F00)[j % 4]
            wl.v_cache[pg, :, j, :] = (0x7F80, 0xFF80, 0x7F00, 0x7FC0)[j % 4]
    return wl


@pytest.mark.parametrize("nodes", [1, 8, 9, 16, 17, 24, 25])
def test_units_that_fill_one_to_four_softmax_warps(nodes):
    """4 heads x nodes rows: one row block warp exactly full, one row over, ...; 64-token pages leave up to 63 dead V rows
    that the live warps alone must clear."""
    wl = W.generate(W.Spec("live", 8, 2, [700 + nodes, 129, 40], [("chain", nodes)] * 3, page_size=64, shuffle_pages=True,
                           seed=700 + nodes, with_logits=False))
    check_attention(fill_dead_slots(wl))
