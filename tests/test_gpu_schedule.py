"""The split-KV schedule, the loads of Q and the merge at group sizes and table widths where their index arithmetic can go
wrong, against the CPU oracle (tolerances as in test_gpu_parity)."""
import numpy as np
import pytest
import torch

from paper_2510_07535_b200 import OwlContext, workloads as W
from paper_2510_07535_b200.runner import DeviceWorkload
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,hkv,nodes", [(1, 2, 64), (3, 2, 43), (5, 1, 51), (6, 2, 1), (7, 1, 36), (9, 1, 28), (12, 2, 10), (128, 1, 2),
                                             (255, 1, 1), (256, 1, 1)])
def test_rows_that_are_not_whole_blocks_of_eight(group, hkv, nodes):
    """Units of 6 to 256 rows, cut into many pieces: eight-row blocks of the merge with rows of two nodes and rows past the
    last, Q rows whose step of eight crosses several nodes or stays within one."""
    wl = W.generate(W.Spec("groups", group * hkv, hkv, [5000 + nodes, 1300], [("tree", nodes, 6)] * 2 if nodes > 1 else [("chain", 1)] * 2,
                           shuffle_pages=True, seed=1200 + group, with_logits=False))
    check_attention(wl)


def test_block_table_too_wide_for_32_bits():
    """A table whose rows could hold 2^24 tiles takes the 64-bit schedule, with the same cuts and so the same results."""
    wl = W.generate(W.Spec("wide", 16, 4, [3000, 40, 900], [("chain", 8), ("tree", 20, 5), ("chain", 1)], page_size=128, shuffle_pages=True,
                           seed=1300, with_logits=False))
    dw = DeviceWorkload.upload(wl)
    ctx = OwlContext(dw.dims)
    dw.attn(ctx)
    out, lse = dw.out.clone(), dw.lse.clone()
    dw.out.zero_(), dw.lse.zero_()
    wide = (1 << 24) // (3 * 4) + 1
    table = torch.full((3, wide), -1, dtype=torch.int32, device="cuda")
    table[:, :dw.block_table.shape[1]] = dw.block_table
    dw.block_table, dw.dims.max_pages_per_seq = table, wide
    dw.attn(ctx)
    assert ctx.owl_get_status() == 0
    assert torch.equal(dw.out, out) and torch.equal(dw.lse, lse)
    assert np.isfinite(dw.out_f32()).all()
    ctx.close()
