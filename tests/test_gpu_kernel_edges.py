"""Kernel branches at the sizes where they can go wrong, against the CPU oracle (tolerances as in test_gpu_parity)."""
import numpy as np
import pytest
import torch

from paper_2510_07535_b200 import OwlContext, make_dims, workloads as W
from test_gpu_parity import check_accept, check_attention
from test_product_plan import ROWS_ON_LANES, SEVERAL_TILES

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


@pytest.mark.parametrize("hkv,ctx", [
    (1, [9000]),                       # one unit cut into 71 pieces: 32 partials per round, three rounds
    (2, [6000] + [20] * 7),            # 12 partials per round, the long units cut into dozens of pieces
    (2, [3000] + [150] * 39),          # 80 units: 4 partials per round, schedule read from global memory
])
def test_merge_rounds_of_partials(hkv, ctx):
    wl = W.generate(W.Spec("merge", 4 * hkv, hkv, ctx, [("tree", 9, 3)] * len(ctx), shuffle_pages=True, seed=800 + len(ctx),
                           with_logits=False))
    check_attention(wl)


@pytest.mark.parametrize("batch,nodes", [(300, 2), (20, 40)])
def test_more_segments_per_cta_than_announced_at_once(batch, nodes):
    """2400 short units over 148 CTAs: 16 segments each, through the eight places the producer announces them in; and
    160 units of 160 rows (both row blocks)."""
    rng = np.random.default_rng(batch)
    # at least 40 keys a row: the 1e-2 of check_attention is meant for outputs well below 1.  A row of a handful of keys is
    # close to a single V row of N(0, 1), up to 4 in magnitude over this many, where rounding the output to bf16 alone is
    # off by up to 2^-9 * 4 = 0.008 and the rounded softmax weights by as much again (0.0112 seen with contexts from 0).
    ctx = [int(x) for x in rng.integers(40, 240, size=batch)]
    hq = 8 if nodes == 2 else 32
    wl = W.generate(W.Spec("segs", hq, 8, ctx, [("chain", nodes)] * batch, shuffle_pages=True, seed=900 + batch, with_logits=False))
    check_attention(wl)


@pytest.mark.parametrize("nodes,vocab", [(1, 50257), (9, 8193), (17, 20001), (33, 128256), (64, 50257)])
def test_scan_items_of_every_size_and_walk_groups(nodes, vocab):
    """Items of 2048 to 8192 floats with ragged rows; 4 to 32 threads per node in the walk."""
    check_accept(W.generate(W.Spec("items", 4, 1, [20] * 3, [("chain", nodes)] * 3, seed=950 + nodes, vocab=vocab)))


@pytest.mark.parametrize("rows,d_in", [(1, 64), (16, 192), (17, 64), (32, 320), (33, 192), (128, 192), (129, 64), (256, 192), (257, 64), (383, 192)])
def test_product_row_padding_and_odd_k_blocks(rows, d_in):
    """The weight-streaming product behind the drafter cell, element by element: rows around the padding to 16 and the
    switch to two column groups (257), one, three and five k-blocks (a stage holds two); one tile per CTA pair.
    Bound: fp32 accumulation of K exact products, K 2^-24 sum_k |h_k| |w_k| per element."""
    d = 4096 + 20
    g = torch.Generator().manual_seed(rows)
    h = torch.randn(rows, d_in, generator=g).bfloat16()
    w = torch.randn(4 * d, d_in, generator=g).bfloat16()
    emb = torch.zeros(rows, d, dtype=torch.bfloat16, device="cuda")
    z, hf = torch.zeros(rows, d, device="cuda"), torch.empty(rows, d, device="cuda")
    ws = torch.full((rows, 4 * d), float("nan"), device="cuda")
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))
    ctx.owl_lstm_cell(h.cuda(), emb, w.cuda(), 0.0, z, hf, None, ws)
    assert ctx.owl_get_status() == 0
    ref = h.double() @ w.double().t()
    bound = d_in * 2.0 ** -24 * (h.double().abs() @ w.double().abs().t())
    assert bool(((ws.cpu().double() - ref).abs() <= bound).all())
    ctx.close()


@pytest.mark.parametrize("rows,d_in,d", SEVERAL_TILES + ROWS_ON_LANES)
def test_product_over_several_tiles_and_in_both_operand_orders(rows, d_in, d):
    """Element by element at the shapes that test_product_plan.py describes.  Bound: fp32 accumulation of K exact products,
    K 2^-24 sum_k |h_k| |w_k| per element."""
    g = torch.Generator(device="cuda").manual_seed(rows + d)
    h = torch.randn(rows, d_in, generator=g, device="cuda").bfloat16()
    w = torch.randn(4 * d, d_in, generator=g, device="cuda").bfloat16()
    emb = torch.zeros(rows, d, dtype=torch.bfloat16, device="cuda")
    z, hf = torch.zeros(rows, d, device="cuda"), torch.empty(rows, d, device="cuda")
    scratch = torch.full((4 * rows * d + 4,), float("nan"), device="cuda")
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))
    ref = h.double() @ w.double().t()
    bound = d_in * 2.0 ** -24 * (h.double().abs() @ w.double().abs().t())
    for first in (0, 1):                                   # scratch that is aligned to 16 bytes, and to 4 only
        ws = scratch[first:first + 4 * rows * d].view(rows, 4 * d)
        ws.fill_(float("nan"))
        ctx.owl_lstm_cell(h, emb, w, 0.0, z, hf, None, ws)
        assert ctx.owl_get_status() == 0
        assert bool(((ws.double() - ref).abs() <= bound).all())
        assert torch.isnan(scratch[first + 4 * rows * d:]).all()
    ctx.close()


def test_small_products_on_two_streams():
    """Products that take a fraction of an SM's shared memory each, of two contexts on two streams at once: every one has to
    have its SMs' tensor memory to itself."""
    rows, d_in, d = 8, 256, 512
    g = torch.Generator().manual_seed(1)
    h = torch.randn(rows, d_in, generator=g).bfloat16()
    w = torch.randn(4 * d, d_in, generator=g).bfloat16()
    hc, wc, emb = h.cuda(), w.cuda(), torch.zeros(rows, d, dtype=torch.bfloat16, device="cuda")
    sides = []
    for _ in range(2):
        sides.append((torch.cuda.Stream(), OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1)), torch.zeros(rows, d, device="cuda"),
                      torch.empty(rows, d, device="cuda"), torch.full((rows, 4 * d), float("nan"), device="cuda")))
    torch.cuda.synchronize()
    for _ in range(50):
        for stream, ctx, z, hf, ws in sides:
            with torch.cuda.stream(stream):
                ctx.owl_lstm_cell(hc, emb, wc, 0.0, z, hf, None, ws)
    torch.cuda.synchronize()
    ref = h.double() @ w.double().t()
    bound = d_in * 2.0 ** -24 * (h.double().abs() @ w.double().abs().t())       # fp32 accumulation of d_in exact products
    for stream, ctx, _, _, ws in sides:
        with torch.cuda.stream(stream):
            assert ctx.owl_get_status() == 0
        assert bool(((ws.cpu().double() - ref).abs() <= bound).all())
        ctx.close()
