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


def _ragged(batch, seed):
    """One tree of 64 nodes among chains of one to five and small trees: units of 4 to 256 rows."""
    rng = np.random.default_rng(seed)
    trees = [("tree", int(rng.integers(2, 13)), 4) if rng.random() < 0.2 else ("chain", int(rng.integers(1, 6))) for _ in range(batch)]
    trees[int(rng.integers(0, batch))] = ("tree", 64, 8)
    lens = [int(x) for x in rng.integers(40, 700, size=batch)]
    lens[int(rng.integers(0, batch))] = 2600
    return W.generate(W.Spec("ragged", 8, 2, lens, trees, shuffle_pages=True, seed=seed, with_logits=False))


@pytest.mark.parametrize("batch", [2, 9, 31, 32, 33, 64, 65, 97, 160])
def test_merge_of_one_large_tree_among_chains(batch):
    """Blocks of rows of sequences of very different sizes: numbered over a warp's lanes, and found by the line's cuts."""
    check_attention(_ragged(batch, 1400 + batch))


@pytest.mark.parametrize("batch,hkv,nodes", [(33, 1, 5), (40, 1, 16), (49, 3, 7), (50, 3, 7), (147, 1, 2), (148, 1, 2)])
def test_merge_by_units_and_by_cuts(batch, hkv, nodes):
    """More than 32 sequences with up to 147 units, which a CTA of the merge goes by, and with more, where it goes by cuts."""
    rng = np.random.default_rng(1600 + batch)
    lens = [int(x) for x in rng.integers(40, 1500, size=batch)]
    check_attention(W.generate(W.Spec("places", 16 * hkv, hkv, lens, [("tree", nodes, 4)] * batch, shuffle_pages=True, seed=1600 + batch,
                                      with_logits=False)))


@pytest.mark.parametrize("batch", [20, 40])
def test_merge_leaves_refused_sequences_out(batch):
    """A sequence without nodes and its neighbour with two roots, in the middle of the batch: the others as without them."""
    wl = _ragged(batch, 1500 + batch)
    dw = DeviceWorkload.upload(wl)
    ctx = OwlContext(dw.dims)
    dw.attn(ctx)
    assert ctx.owl_get_status() == 0
    out, lse = dw.out.clone(), dw.lse.clone()
    offs = wl.node_offsets.copy()
    b = next(i for i in range(batch // 2, batch) if 1 <= offs[i + 1] - offs[i] <= 8 and offs[i + 2] - offs[i + 1] <= 8)
    rows = slice(int(offs[b]), int(offs[b + 2]))
    dw.node_offsets[b + 1] = int(offs[b])
    dw.out.fill_(7.0), dw.lse.fill_(7.0)
    dw.attn(ctx)
    assert ctx.owl_get_status() == -4
    out[rows], lse[rows] = 7.0, 7.0
    # the cuts move with the units that are gone: another order of the same fp32 sums, then one bf16 rounding of values below 4
    assert float((dw.out.float() - out.float()).abs().max()) <= 2.0 ** -7 and float((dw.lse - lse).abs().max()) <= 1e-4
    assert torch.equal(dw.out[rows], out[rows]) and torch.equal(dw.lse[rows], lse[rows])
    ctx.close()
