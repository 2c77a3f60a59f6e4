"""The producers either side of the verify step on the GPU, through the C ABI, against the CPU oracle: acceptance
straight from hidden states (LM-head product with the arg-max in its epilogue) and the drafter's LSTM cell (Eq. 1-8)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_07535_b200 import OwlContext, make_dims, workloads as W
from paper_2510_07535_b200.binding import owl_lstm_alpha

pytestmark = pytest.mark.gpu

DEV = "cuda"
dev_i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)
dev_bf16 = lambda bits: torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).to(DEV).view(torch.bfloat16)


def _normal_bits(seed, shape, scale=1.0):
    ss = np.random.SeedSequence(seed)
    return W.normal_bf16(ss, int(np.prod(shape)), scale=scale).reshape(shape)


def _oracle_rows(hidden, weight, chunk=16384):
    """Per row: the oracle's arg-max, and the slack tau_row within which fp32 accumulation may rank two logits either
    way, from the oracle's fp64 logits computed vocabulary chunk by chunk (bounded memory)."""
    N, K = hidden.shape
    V = weight.shape[0]
    logits = np.empty((N, V))
    absmax = np.zeros(N)
    ha = np.abs(oracle.decode16(hidden, "bf16").reshape(N, K))
    for v0 in range(0, V, chunk):
        w = weight[v0:v0 + chunk]
        logits[:, v0:v0 + len(w)] = oracle.lm_head_logits(hidden, w)
        absmax = np.maximum(absmax, (ha @ np.abs(oracle.decode16(w, "bf16").reshape(len(w), K)).T).max(axis=1))
    tau = 2.0 * K * 2.0 ** -24 * absmax
    return logits, tau


def _lm_head_case(ctx, seed, trees, K, V, plant=0.7):
    rng = np.random.default_rng(seed)
    parents = [W.chain_parents(t[1]) if t[0] == "chain" else W.random_tree_parents(rng, t[1], t[2]) for t in trees]
    counts = np.array([len(p) for p in parents])
    offs = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    par = np.concatenate(parents).astype(np.int32)
    N, B = len(par), len(trees)
    hidden = _normal_bits(seed, (N, K))
    weight = _normal_bits(seed + 1, (V, K), scale=1.0 / np.sqrt(K))
    logits, tau = _oracle_rows(hidden, weight)
    am_ref = oracle.row_argmax(logits.astype(np.float32))          # (fp32 rounding of fp64 logits keeps the order up to ties)
    am_ref = np.argmax(logits, axis=1).astype(np.int32)            # first maximum of the fp64 logits
    # drafted tokens: with probability `plant` the target's own continuation of the parent, else another token
    tok = rng.integers(0, V, size=N).astype(np.int32)
    for b in range(B):
        for i in range(1, counts[b]):
            if rng.random() < plant:
                tok[offs[b] + i] = am_ref[offs[b] + par[offs[b] + i]]
    d = make_dims(batch=B, total_nodes=N, max_nodes=int(counts.max()), vocab=V)
    alen = torch.full((B,), -3, dtype=torch.int32, device=DEV); path = torch.full((B, 64), -3, dtype=torch.int32, device=DEV)
    bonus = torch.full((B,), -3, dtype=torch.int32, device=DEV); am = torch.full((N,), -3, dtype=torch.int32, device=DEV)
    hd, wd = dev_bf16(hidden), dev_bf16(weight)
    for _ in range(2):                                             # twice: the keys are cleared by the call itself
        ctx.owl_lm_head_accept(d, hd, wd, dev_i32(tok), dev_i32(offs), dev_i32(par), alen, path, bonus, am)
        assert ctx.owl_get_status() == 0
        am_gpu = am.cpu().numpy()
        rows = np.arange(N)
        # tolerance-aware arg-max: the chosen logit is within tau_row of the row maximum; lowest index on exact ties
        assert np.all(logits[rows, am_gpu] >= logits.max(axis=1) - tau), np.abs(logits[rows, am_gpu] - logits.max(axis=1)).max()
        gap = np.sort(logits, axis=1)[:, -1] - np.sort(logits, axis=1)[:, -2]
        clear = gap > tau
        assert clear.mean() > 0.8          # the test keeps its power: most rows have an unambiguous arg-max
        np.testing.assert_array_equal(am_gpu[clear], am_ref[clear])
        # the walk is integer work: bit for bit what the oracle's walk gives on the same arg-max
        r_alen, r_path, r_bonus = oracle.accept_from_argmax(offs, par, tok, am_gpu, 64)
        np.testing.assert_array_equal(alen.cpu().numpy(), r_alen)
        np.testing.assert_array_equal(path.cpu().numpy(), r_path)
        np.testing.assert_array_equal(bonus.cpu().numpy(), r_bonus)
        if clear.all():
            o_alen, o_path, o_bonus = oracle.accept_from_argmax(offs, par, tok, am_ref, 64)
            np.testing.assert_array_equal(alen.cpu().numpy(), o_alen)
            np.testing.assert_array_equal(bonus.cpu().numpy(), o_bonus)
        alen.fill_(-3); am.fill_(-3)
    return r_alen


@pytest.mark.parametrize("trees,K,V", [
    ([("chain", 8)], 128, 1000),                                    # 8 rows, tiles of 16 weight rows, the last one ragged
    ([("tree", 20, 4), ("chain", 3)], 64, 129),                     # a single k-block; a tile of one weight row
    ([("tree", 64, 8)] * 3 + [("chain", 8)], 256, 5000),            # 200 rows on the lanes, one tile of 80 weight rows
    ([("tree", 64, 8)] * 5, 512, 3000),                             # 320 rows in two groups on the lanes, tiles of 48
    ([("tree", 32, 6)], 4096, 20000),                               # the real hidden width: 64 k-blocks, two rounds (144 + 128)
    ([("tree", 64, 8)] * 3, 64, 40000),                             # 192 rows on the lanes, three rounds (192 + 2 x 176), half of each stage past K
    ([("tree", 64, 8)] * 5, 64, 20000),                             # 320 rows in two groups, two rounds (144 + 128), one accumulator buffer
    ([("chain", 5)], 64, 16),                                       # the whole vocabulary is one tile of 16 on one CTA pair
    ([("tree", 64, 8)] * 2 + [("chain", 2)], 128, 16),              # 130 rows on the lanes of one CTA pair: one stage, one tile of 16
    ([("tree", 64, 8)] * 4, 128, 1000),                             # 256 rows on the lanes: 63 pairs with a tile of 16 each
    ([("tree", 40, 6)] * 4, 384, 40000),                            # 160 rows, weights on the lanes: three rounds (192 + 2 x 176), three stages per tile
    ([("tree", 64, 8)] * 6, 128, 40000),                            # 384 rows in two groups on the lanes, three rounds, two stages per tile
    ([("tree", 64, 8)] * 4 + [("chain", 1)], 256, 2000),            # 257 rows: two groups of 144
])
def test_lm_head_accept_small(trees, K, V):
    ctx = OwlContext(make_dims(batch=8, total_nodes=384, max_nodes=64, vocab=V))
    alen = _lm_head_case(ctx, 1000 + K + V, trees, K, V)
    assert alen.max() > 1
    ctx.close()


@pytest.mark.parametrize("trees,K,V", [
    ([("tree", 64, 8)] * 5, 4096, 12000),                           # 320 rows at a real hidden width: 64 stages of one k-block through a ring of six
    ([("tree", 64, 8)] * 2, 1024, 5000),                            # rows of A on the lanes (tiles of 80 weight rows): 128 rows
    ([("tree", 64, 8)] * 4, 448, 40000),                            # ... 256 rows, three rounds, seven k-blocks
    ([("tree", 64, 8)] * 4 + [("chain", 1)], 192, 5000),            # ... 257 rows in two groups
    ([("tree", 64, 8)] * 6, 1024, 2000),                            # ... 384 rows, tiles of 32
])
def test_lm_head_accept_in_both_operand_orders(trees, K, V):
    ctx = OwlContext(make_dims(batch=8, total_nodes=384, max_nodes=64, vocab=V))
    alen = _lm_head_case(ctx, 2000 + K + V, trees, K, V)
    assert alen.max() > 1
    ctx.close()


def test_rows_on_lanes_ties_infinities_and_nan():
    """100 rows against 5000 weight rows: the arg-max of equal logits is the lowest index (equal weight rows in one tile, in
    two tiles of a pair's CTAs and in tiles of different pairs), -inf everywhere gives 0, and NaN never wins."""
    N, K, V = 100, 64, 5000
    hidden = torch.zeros(N, K, device=DEV, dtype=torch.bfloat16)
    weight = torch.zeros(V, K, device=DEV, dtype=torch.bfloat16)
    hidden[:, 0] = 1.0
    weight[:, 0] = -1.0
    want = []
    for i in range(N - 2):                              # row i looks at feature 1 + i % 32: equal logits at three columns
        f, cols = 1 + i % 32, sorted({7 + 5 * (i % 32), 47 + 5 * (i % 32), 2600 + 61 * (i % 32)})
        hidden[i, f] = 2.0
        weight[cols, f] = 3.0
        want.append(cols[0])
    weight[3, 40], hidden[10, 40] = float("nan"), 1.0   # column 3 is NaN for every row
    hidden[N - 2, 0] = float("inf")
    want += [0, 0]                                      # -inf (and NaN in column 3) everywhere; all -1: the first
    d = make_dims(batch=N, total_nodes=N, max_nodes=1, vocab=V)
    ctx = OwlContext(d)
    outs = [torch.zeros(N, dtype=torch.int32, device=DEV), torch.zeros(N, 64, dtype=torch.int32, device=DEV)] + \
           [torch.zeros(N, dtype=torch.int32, device=DEV) for _ in range(2)]
    tok = torch.zeros(N, dtype=torch.int32, device=DEV)
    ctx.owl_lm_head_accept(d, hidden, weight, tok, None, tok - 1, *outs)
    assert ctx.owl_get_status() == 0
    assert outs[3].cpu().tolist() == want
    ctx.close()


def test_lm_head_accept_calls_of_different_sizes_on_one_context():
    """The row keys live in two sets that alternate between calls, each cleared as a whole by the call before: a
    200-row call, an 8-row call, a 200-row call and a 23-row call through one context (two launches each inside
    the helper, so every set is reused after a larger and after a smaller call) all match the oracle."""
    ctx = OwlContext(make_dims(batch=8, total_nodes=384, max_nodes=64, vocab=5000))
    big = [("tree", 64, 8)] * 3 + [("chain", 8)]
    for k, trees in enumerate([big, [("chain", 8)], big, [("tree", 20, 4), ("chain", 3)]]):
        _lm_head_case(ctx, 4000 + k, trees, 128, 5000)
    ctx.close()


@pytest.mark.parametrize("captured", [1, 2, 3])
def test_lm_head_accept_replayed_from_a_graph_on_new_inputs(captured):
    """A graph of one, two or three calls, replayed on hidden states that shrink from replay to replay (whatever is left of
    an earlier replay's arg-max keys would win), between calls made directly on the same context."""
    N, K, V = 12, 128, 3000
    d = make_dims(batch=2, total_nodes=N, max_nodes=6, vocab=V)
    ctx = OwlContext(d)
    par, tok = dev_i32(np.tile(W.chain_parents(6), 2)), torch.zeros(N, dtype=torch.int32, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(7)
    weight = torch.randn(V, K, generator=g, device=DEV, dtype=torch.bfloat16)
    fresh = [torch.randn(N, K, generator=g, device=DEV).mul_(4.0 ** -r).to(torch.bfloat16) for r in range(8)]
    hidden = fresh[0].clone()
    outs = [[torch.zeros(2, dtype=torch.int32, device=DEV), torch.zeros(2, 64, dtype=torch.int32, device=DEV),
             torch.zeros(2, dtype=torch.int32, device=DEV), torch.zeros(N, dtype=torch.int32, device=DEV)] for _ in range(captured)]
    call = lambda o: ctx.owl_lm_head_accept(d, hidden, weight, tok, None, par, *o)
    call(outs[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for o in outs:
            call(o)
    for r, h in enumerate(fresh):
        hidden.copy_(h)
        want = torch.argmax(h.double() @ weight.double().t(), dim=1).int()
        for o in outs:
            o[3].fill_(-1)
        graph.replay()
        assert all(torch.equal(o[3], want) for o in outs), r
        if r % 3 == 1:
            outs[0][3].fill_(-1)
            call(outs[0])
            assert torch.equal(outs[0][3], want), r
    assert ctx.owl_get_status() == 0
    del graph
    ctx.close()


def test_lm_head_accept_full_vocabulary():
    """The 8B shape's head: hidden 4096, vocabulary 128256 (7 rounds of tiles over 74 CTA pairs), a 32-node tree."""
    ctx = OwlContext(make_dims(batch=1, total_nodes=32, max_nodes=32, vocab=W.VOCAB))
    _lm_head_case(ctx, 77, [("tree", 32, 6)], 4096, W.VOCAB)
    ctx.close()


def test_lm_head_accept_full_vocabulary_on_cta_pairs():
    """Four 64-node trees (256 rows, on the lanes): seven rounds of tiles of 256 and 240 weight rows over 74 CTA pairs, both
    accumulator buffers in turn."""
    ctx = OwlContext(make_dims(batch=4, total_nodes=256, max_nodes=64, vocab=W.VOCAB))
    _lm_head_case(ctx, 78, [("tree", 64, 8)] * 4, 4096, W.VOCAB)
    ctx.close()


def test_lm_head_accept_errors():
    ctx = OwlContext(make_dims(batch=8, total_nodes=400, max_nodes=64, vocab=1000))
    one = torch.zeros(400, dtype=torch.int32, device=DEV)
    hid = torch.zeros((400, 96), dtype=torch.bfloat16, device=DEV)
    wt = torch.zeros((1000, 96), dtype=torch.bfloat16, device=DEV)
    n0 = ctx.launch_count()
    d = make_dims(batch=2, total_nodes=16, max_nodes=8, vocab=1000)
    assert ctx.owl_lm_head_accept(d, hid[:16], wt, one, None, one, one, one, one, check=False) == -2      # 96 is no multiple of 64
    d = make_dims(batch=8, total_nodes=400, max_nodes=64, vocab=1000)
    assert ctx.owl_lm_head_accept(d, hid[:, :64].contiguous(), wt[:, :64].contiguous(), one, None, one, one, one, one, check=False) in (-2, -7)
    d = make_dims(batch=2, total_nodes=16, max_nodes=8, vocab=1000)
    assert ctx.owl_lm_head_accept(d, None, wt, one, None, one, one, one, one, check=False) == -1
    assert ctx.launch_count() == n0
    ctx.close()


# ----------------------------------------------------------------------------- drafter cell

def _cell_case(ctx, seed, M, d_in, d, affine, steps=1, z_mean=0.0):
    rng = np.random.default_rng(seed)
    hb = _normal_bits(seed, (M, d_in))
    eb = _normal_bits(seed + 1, (M, d))
    wb = _normal_bits(seed + 2, (4 * d, d_in), scale=1.0 / np.sqrt(d_in))
    alpha = 0.8 if d < 1000 else owl_lstm_alpha(8, d) * 100          # large enough for the embedding to matter
    ln_c = (rng.uniform(0.5, 1.5, d).astype(np.float32), rng.normal(0, 0.2, d).astype(np.float32)) if affine else (None, None)
    ln_z = (rng.uniform(0.5, 1.5, d).astype(np.float32), rng.normal(0, 0.2, d).astype(np.float32)) if affine else (None, None)
    t = lambda a: None if a is None else torch.from_numpy(a).to(DEV)
    z = (z_mean + rng.standard_normal((M, d))).astype(np.float32) if steps == 1 else np.zeros((M, d), np.float32)
    zd = torch.from_numpy(z.copy()).to(DEV)
    hf = torch.zeros((M, d), dtype=torch.float32, device=DEV)
    hb16 = torch.zeros((M, d), dtype=torch.bfloat16, device=DEV)
    ws = torch.empty((M, 4 * d), dtype=torch.float32, device=DEV)
    h_dev = dev_bf16(hb)
    z_ref = z.astype(np.float64)
    h_bits = hb
    for step in range(steps):
        ctx.owl_lstm_cell(h_dev, dev_bf16(eb), dev_bf16(wb), alpha, zd, hf, hb16, ws, (t(ln_c[0]), t(ln_c[1])), (t(ln_z[0]), t(ln_z[1])))
        assert ctx.owl_get_status() == 0
        h_ref, z_ref = oracle.lstm_cell(h_bits, eb, wb.reshape(4, d, d_in), z_ref, alpha, ln_c, ln_z)
        ez = np.abs(zd.cpu().numpy() - z_ref).max()
        eh = np.abs(hf.cpu().numpy() - h_ref).max()
        assert ez <= 2e-3 and eh <= 2e-3, (step, ez, eh)
        hb_ref = hb16.float().cpu().numpy()
        assert np.all(np.abs(hb_ref - h_ref) <= 2e-3 + 2.0 ** -8 * np.abs(h_ref))
        if steps > 1:
            # recurrence (d_in == d): the next step consumes the bf16 h' the device produced; the oracle follows the same bits
            assert d_in == d
            h_bits = hb16.view(torch.int16).cpu().numpy().view(np.uint16)
            h_dev = hb16.clone()
            z_ref = zd.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("M,d_in,d,affine", [
    (1, 64, 64, False),
    (5, 128, 260, True),            # 1040 weight rows: 65 pairs with a tile of 16 each
    (130, 256, 512, True),          # rows on the lanes
    (300, 64, 128, False),          # two groups of rows on the lanes
    (2, 64, 4, True),               # fewer columns than CTAs in a row's cluster: half of them hold none
    (1, 64, 16384, True),           # the widest cell: four columns per thread, four rounds of product tiles
    (256, 128, 4096, False),        # all 128 lanes of both CTAs hold rows; a tile of 224
    (129, 384, 36, True),           # rows on the lanes; 144 weight rows in all
    (300, 256, 512, True),          # two groups of rows on the lanes, tiles of 32
])
def test_lstm_cell_small(M, d_in, d, affine):
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))
    _cell_case(ctx, 500 + M, M, d_in, d, affine)
    ctx.close()


def test_lstm_cell_state_with_a_large_mean():
    """z ~ +-300 + N(0, 1): z' = z g^f + ... is of the order of a hundred with a non-zero mean, so the second layer
    normalisation works far from the origin (the kernel takes its variance about the mean: per-CTA means and sums of
    squared deviations, combined).  Same tolerance as everywhere; the oracle carries the same z in fp64."""
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))
    _cell_case(ctx, 950, 3, 128, 4096, True, z_mean=300.0)
    _cell_case(ctx, 951, 130, 128, 260, False, z_mean=-300.0)
    ctx.close()


def test_lstm_cell_paper_width_and_recurrence():
    """d_in = 4096 -> d = 12288 (Section 4.1), ten drafter states; then three recurrent steps at d_in = d = 1024."""
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))
    _cell_case(ctx, 900, 10, 4096, 12288, True)
    _cell_case(ctx, 901, 4, 1024, 1024, False, steps=3)
    ctx.close()


def test_lstm_cell_errors_and_alpha():
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))
    assert abs(owl_lstm_alpha(8, 12288) - oracle.lstm_alpha(8, 12288)) < 1e-15
    h = torch.zeros((2, 96), dtype=torch.bfloat16, device=DEV); e = torch.zeros((2, 64), dtype=torch.bfloat16, device=DEV)
    w = torch.zeros((256, 96), dtype=torch.bfloat16, device=DEV); f = torch.zeros((2, 256), dtype=torch.float32, device=DEV)
    n0 = ctx.launch_count()
    assert ctx.owl_lstm_cell(h, e, w, 0.5, f[:, :64].contiguous(), f[:, :64].contiguous(), None, f, check=False) == -2   # d_in = 96
    h64 = torch.zeros((2, 64), dtype=torch.bfloat16, device=DEV); w64 = torch.zeros((256, 64), dtype=torch.bfloat16, device=DEV)
    assert ctx.owl_lstm_cell(h64, e, w64, 0.5, f[:, :64].contiguous(), None, None, f, check=False) == -1                 # no output
    assert ctx.launch_count() == n0
    ctx.close()
