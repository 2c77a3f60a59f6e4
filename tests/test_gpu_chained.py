"""Calls queued one behind the other with no host synchronisation between them, each on what the one before left in place: the
kernels that read inputs before their dependency wait have to see it.  Bit for bit what the same calls give one at a time,
and those against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_07535_b200 import OwlContext, make_dims, workloads as W
from test_gpu_loop import bits_of, dev_bf16, dev_i32

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.mark.parametrize("rows,d_in,d", [(10, 128, 260),      # 33 columns of z per CTA: neighbours share lines
                                         (3, 320, 320),       # h' fed back
                                         (20, 1024, 1024)])
def test_cells_in_a_chain(rows, d_in, d):
    steps = 12
    g = torch.Generator().manual_seed(rows)
    rand = lambda *shape, scale=1.0: (torch.randn(*shape, generator=g) * scale).to(DEV)
    h0, w = rand(rows, d_in).bfloat16(), rand(4 * d, d_in, scale=d_in ** -0.5).bfloat16()
    embs = [rand(rows, d).bfloat16() for _ in range(steps)]
    ln = [(1 + rand(d, scale=0.1), rand(d, scale=0.1)) for _ in range(2)]
    ws = torch.empty(rows, 4 * d, device=DEV)
    ctx = OwlContext(make_dims(batch=1, total_nodes=1, max_nodes=1))

    def run(chained):
        z, emb = torch.zeros(rows, d, device=DEV), torch.zeros(rows, d, dtype=torch.bfloat16, device=DEV)
        hf, hb = torch.zeros(steps, rows, d, device=DEV), torch.zeros(steps, rows, d, dtype=torch.bfloat16, device=DEV)
        h = h0
        for i in range(steps):
            if i % 3 == 0:
                emb.copy_(embs[i])           # written right in front of a call; otherwise two cells are neighbours
            z_before = None if chained else z.cpu().numpy().astype(np.float64)
            ctx.owl_lstm_cell(h, emb, w, 0.3, z, hf[i], hb[i], ws, ln_c=ln[0], ln_z=ln[1])
            if not chained:
                torch.cuda.synchronize()
                h_ref, z_ref = oracle.lstm_cell(bits_of(h), bits_of(emb), bits_of(w).reshape(4, d, d_in), z_before, 0.3,
                                                *[tuple(t.cpu().numpy() for t in pair) for pair in ln])
                assert np.abs(z.cpu().numpy() - z_ref).max() <= 2e-3 and np.abs(hf[i].cpu().numpy() - h_ref).max() <= 2e-3
            if d_in == d:
                h = hb[i]
        assert ctx.owl_get_status() == 0
        return hf, hb, z

    one_at_a_time = run(False)
    for _ in range(3):
        for got, want in zip(run(True), one_at_a_time):
            assert torch.equal(got, want)
    ctx.close()


@pytest.mark.parametrize("lens,kinds", [([700], [("tree", 30)]), ([130, 45, 900], [("chain", 7), ("tree", 30), ("tree", 12)])])
def test_rounds_in_a_chain(lens, kinds):
    """Prepare on a routed batch, attention, acceptance with the [SPEC] leaf, commit: lengths, cache and prepared trees only
    ever on the device, ten rounds in a row."""
    rounds, hq, hkv, page, vocab = 10, 8, 2, 16, 3000
    rng = np.random.default_rng(sum(lens))
    B = len(lens)
    parents = [W.chain_parents(n) if kind == "chain" else W.random_tree_parents(rng, n, 8) for kind, n in kinds]
    counts = [n for _, n in kinds]
    full = [n if kind == "chain" else 2 * n for kind, n in kinds]
    offs = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    par = np.concatenate(parents).astype(np.int32)
    tok = np.concatenate([rng.permutation(vocab - 1)[:n] for n in counts]).astype(np.int32)
    route = np.array([0 if kind == "chain" else 2 for kind, _ in kinds], np.int32)
    N, M = sum(counts), sum(full)
    pages = (max(lens) + 9 * rounds + 64) // page + 1
    table = rng.permutation(B * pages).astype(np.int32).reshape(B, pages)
    bits = lambda *shape, scale=1.0: W.f32_to_bf16_bits((rng.standard_normal(shape) * scale).astype(np.float32))
    k0, v0, q = bits(B * pages, hkv, page, 128), bits(B * pages, hkv, page, 128), bits(M, hq, 128, scale=128 ** -0.5)
    r_offs, r_par, r_tok, _, _ = oracle.prepare_hybrid(offs, par, tok, np.array(lens, np.int32), route, vocab - 1)
    logits = rng.standard_normal((M, vocab)).astype(np.float32)
    for b in range(B):
        for i in range(1, counts[b]):
            if rng.random() < 0.7:
                logits[r_offs[b] + r_par[r_offs[b] + i], r_tok[r_offs[b] + i]] += 10
    pd = make_dims(batch=B, total_nodes=N, max_nodes=max(counts))
    d = make_dims(batch=B, total_nodes=M, max_nodes=max(full), num_q_heads=hq, num_kv_heads=hkv, page_size=page, max_pages_per_seq=pages,
                  num_pages=B * pages, vocab=vocab)
    ctx = OwlContext(d)
    inputs = [dev_i32(a) for a in (offs, par, tok, route, table)]
    offs_d, par_d, tok_d, route_d, table_d = inputs
    q_d, lg = dev_bf16(q), torch.from_numpy(logits).to(DEV)

    def run(chained):
        k, v, ld = dev_bf16(k0), dev_bf16(v0), dev_i32(lens)
        prep = [torch.zeros(B + 1, dtype=torch.int32, device=DEV)] + [torch.zeros(2 * N, dtype=torch.int32, device=DEV) for _ in range(4)]
        out, lse = torch.zeros(rounds, M, hq, 128, dtype=torch.bfloat16, device=DEV), torch.zeros(rounds, M, hq, device=DEV)
        small = torch.zeros(rounds, 3, B, dtype=torch.int32, device=DEV)
        path = torch.zeros(rounds, B, 64, dtype=torch.int32, device=DEV)
        for i in range(rounds):
            ctx.owl_prepare_hybrid(pd, offs_d, par_d, tok_d, ld, route_d, vocab - 1, *prep)
            ctx.owl_verify_attn(d, q_d, k, v, table_d, ld, prep[0], prep[1][:M], out[i], lse[i])
            ctx.owl_tree_accept_spec(d, lg, prep[2][:M], prep[0], prep[1][:M], small[i, 0], path[i], small[i, 1], small[i, 2], None)
            if not chained:
                torch.cuda.synchronize()
                ref_out, ref_lse = oracle.verify_attn(q, bits_of(k), bits_of(v), table, ld.cpu().numpy(), r_offs, r_par, 1.0)
                assert np.abs(out[i].float().cpu().numpy() - ref_out).max() <= 1e-2 and np.abs(lse[i].cpu().numpy() - ref_lse).max() <= 1e-3
            ctx.owl_kv_commit(d, k, v, table_d, ld, prep[0], small[i, 0], path[i])
        assert ctx.owl_get_status() == 0
        return out, lse, small, path, prep[4], ld, k, v

    one_at_a_time = run(False)
    alen, r_path, bonus, _ = oracle.tree_accept(logits, r_tok, r_offs, r_par, 64)
    assert one_at_a_time[5].cpu().tolist() == (np.array(lens) + rounds * alen).tolist()
    assert np.array_equal(one_at_a_time[3][-1].cpu().numpy(), r_path) and np.array_equal(one_at_a_time[2][-1, 1].cpu().numpy(), bonus)
    for _ in range(3):
        for got, want in zip(run(True), one_at_a_time):
            assert torch.equal(got, want)
    ctx.close()
