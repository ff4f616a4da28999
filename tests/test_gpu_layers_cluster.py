"""Decode passes in clusters of 16 CTAs. Rows inside one cluster (layers_cluster.cuh), at the edges of its rows per cluster (8, 16, 32, 48,
64 times the seven clusters of the device); up to 16 rows at d = 1024 with the weights split between the clusters (layers_split.cuh; one, two
and three layers): logits, tokens and cache against the kernel-per-operation path fed the
same tokens, rows of the batch against the oracle, equal and per-sample positions, all cache types."""
import numpy as np
import pytest
import torch

import srm_inputs as I
from helpers import custom_shape, oracle_for, rel_err_rows, top2_margin

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,d,layers,state_dtype,ragged", [
    (1, 1024, 3, "fp32", False), (2, 1024, 1, "fp16", False), (8, 1024, 2, "fp32", True), (9, 1024, 3, "bf16", False), (16, 1024, 3, "fp16", True),
    (17, 1024, 3, "fp16", False), (25, 1024, 2, "fp32", False), (32, 1024, 3, "fp32", True), (33, 1024, 3, "bf16", False),
    (111, 512, 3, "fp32", False), (113, 512, 3, "fp16", True), (224, 512, 3, "bf16", False), (225, 512, 3, "fp32", True), (336, 512, 3, "fp16", False),
    (337, 512, 3, "fp32", False), (448, 512, 3, "fp32", True), (449, 512, 3, "fp32", False), (56, 1024, 3, "fp32", True),
    (57, 1024, 3, "fp32", False), (100, 1024, 3, "bf16", True), (112, 1024, 3, "fp16", False)])
def test_rows_in_clusters_agree_with_the_kernel_per_operation_path(B, d, layers, state_dtype, ragged):
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=layers, d_model=d, vocab=2048, n_ctx=24, dtype="bf16", seed=19)
    W = I.make_weights(shape)
    rng = np.random.default_rng(B)
    n = 5
    prompts_np = rng.integers(0, shape.vocab, size=(B, n)).astype(np.int32)
    lens_np = rng.integers(1, n + 1, size=B).astype(np.int32) if ragged else np.full(B, n, np.int32)
    fed = torch.from_numpy(rng.integers(0, shape.vocab, size=(3, B)).astype(np.int32)).to(DEV)
    prompts, lens = torch.from_numpy(prompts_np).to(DEV), torch.from_numpy(lens_np).to(DEV)
    g = P.Sampling("greedy")
    outs = []
    for flags in (P.FLAG_NO_SMALL_BATCH, 0):
        m = P.SRM(shape, W, device=DEV, flags=flags, state_dtype=state_dtype)
        st, ws = m.new_state(B), m.new_workspace(B, n, prefill_samples=B)
        one_kernel = "split" if d == 1024 and B <= 16 else "clusters" if B <= (112 if d == 1024 else 448) else "layers"
        assert m.decode_route(B, ws) == ("kernels" if flags else one_kernel)
        m.prefill_ragged(st, prompts, lens, g, ws) if ragged else m.prefill(st, prompts, g, ws)
        lgs, toks = [], []
        for k in range(3):
            tok, lg = m.decode_step(st, fed[k], g, k + 1, ws, want_logits=True)
            lgs.append(lg.cpu().numpy())
            toks.append(tok.cpu().numpy())
        assert st.status() == 0
        outs.append((np.stack(lgs), np.stack(toks), st.cache().cpu().float().numpy()))
    (lg_a, tok_a, S_a), (lg_b, tok_b, S_b) = outs
    # Sums in another order flip roundings of bf16 activations, 2^-8 of the value each. Were half of them flipped, a
    # layer would move its output by 2^-9 of its scale, all layers by 2^-9 sqrt(layers); five standard deviations of that:
    tol = 5 * 2.0 ** -9 * layers ** 0.5
    assert rel_err_rows(lg_b, lg_a) < tol and rel_err_rows(S_b, S_a) < tol
    assert np.all(top2_margin(lg_a)[tok_a != tok_b] < 2e-2)
    orc = oracle_for(shape, W)
    for b in (0, B // 2, B - 1):
        lo, state = orc.forward_parallel(prompts_np[b:b + 1, :lens_np[b]])
        for k in range(3):
            lo, state = orc.decode_step(state, fed[k, b:b + 1].cpu().numpy(), int(lens_np[b]) + k)
            assert rel_err_rows(lg_b[k][b:b + 1], lo) < 3e-2


def test_a_row_has_the_same_bits_in_any_pass():
    """300 rows at d = 512 in one pass, in passes of 100 and backwards: bit-equal (instances of the kernel for 16 and 48 rows)."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=2, d_model=512, vocab=1024, n_ctx=16, dtype="bf16", seed=20)
    W = I.make_weights(shape)
    B = 300
    toks = torch.from_numpy(np.random.default_rng(4).integers(0, shape.vocab, size=(4, B)).astype(np.int32)).to(DEV)
    g = P.Sampling("greedy")
    res = []
    for order, chunk in ((1, B), (1, 100), (-1, B)):
        m = P.SRM(shape, W, device=DEV)
        st, ws = m.new_state(B), m.new_workspace(chunk)
        lgs = [m.decode_step(st, (t if order > 0 else t.flip(0)).contiguous(), g, k + 1, ws, want_logits=True)[1].clone() for k, t in enumerate(toks)]
        assert st.status() == 0
        res.append([lg if order > 0 else lg.flip(0) for lg in lgs] + [st.cache() if order > 0 else st.cache().flip(1)])
    for r in res[1:]:
        for x, y in zip(res[0], r):
            assert torch.equal(x, y)


@pytest.mark.parametrize("B,d,state_dtype", [(448, 512, "fp32"), (256, 512, "fp16"), (17, 1024, "fp32"), (112, 1024, "fp32")])
def test_thousands_of_passes_give_the_same_bits(B, d, state_dtype):
    """The kernel's exchanges through shared memory, whatever their timing: the same 500 steps again and again (4000 passes)."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=4, d_model=d, vocab=2048, n_ctx=504, dtype="bf16", seed=22)
    m = P.SRM(shape, I.make_weights(shape), device=DEV, state_dtype=state_dtype)
    tok = torch.from_numpy(np.random.default_rng(B).integers(0, shape.vocab, size=(B, 1)).astype(np.int32)).to(DEV)
    g = P.Sampling("greedy")
    st, ws = m.new_state(B), m.new_workspace(B, 1, prefill_samples=B)
    first = None
    for _ in range(8):
        st.reset()
        m.prefill(st, tok, g, ws)
        out, cache = m.generate(st, 500, 1, g, ws).clone(), st.cache().clone()
        first = first or (out, cache)
        assert torch.equal(out, first[0]) and torch.equal(cache, first[1])
    assert st.status() == 0


@pytest.mark.parametrize("B,d,vocab", [(1, 512, 1000), (7, 512, 2056), (16, 512, 128), (64, 512, 8000), (113, 512, 136), (225, 512, 1920),
                                       (337, 512, 5000), (448, 512, 2048), (1, 1024, 8000), (2, 1024, 136), (9, 1024, 4488), (16, 1024, 32000)])
def test_selection_in_the_same_kernel_equals_selection_from_the_logits(B, d, vocab):
    """Greedy steps of one launch: vocabularies that leave ranks (or CTAs) without a tile, end inside a tile, give unequal numbers of
    tiles. The same products in two orders of addition (at most 1024 terms, fp32): ids must agree where the two largest logits differ by more than
    2^-20 of the largest, sixteen times the rounding of one addition."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=2, d_model=d, vocab=vocab, n_ctx=16, dtype="bf16", seed=21)
    m = P.SRM(shape, I.make_weights(shape), device=DEV)
    toks = torch.from_numpy(np.random.default_rng(B).integers(0, vocab, size=(3, B)).astype(np.int32)).to(DEV)
    g = P.Sampling("greedy")
    a, b, ws = m.new_state(B), m.new_state(B), m.new_workspace(B)
    strict = 0
    for k in range(3):
        n0 = P.SRM.kernel_launches()
        tok_a = m.decode_step(a, toks[k], g, k + 1, ws)
        assert P.SRM.kernel_launches() - n0 == 1
        tok_b, lg = m.decode_step(b, toks[k], g, k + 1, ws, want_logits=True)
        lg = lg.cpu().numpy()
        clear = top2_margin(lg) > 2.0 ** -20 * np.abs(lg).max(-1)
        strict += clear.mean() / 3
        assert np.array_equal(tok_a.cpu().numpy()[clear], tok_b.cpu().numpy()[clear])
        assert torch.equal(a.last_token(), tok_a)
    assert strict > 0.9 and a.status() == 0 and b.status() == 0 and torch.equal(a.cache(), b.cache())


@pytest.mark.parametrize("B,vocab", [(1, 8), (1, 128), (5, 1000), (7, 1920), (40, 8), (112, 136), (113, 1912), (448, 264)])
def test_vocabularies_that_leave_ranks_without_a_tile(B, vocab):
    """Greedy steps of one launch at d = 512, a thousand of them: ranks of a cluster without vocabulary rows, with and without rows of the batch,
    send their part of the selection when its receivers have done with the last layer, not before."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=1, d_model=512, vocab=vocab, n_ctx=1008, dtype="bf16", seed=23)
    m = P.SRM(shape, I.make_weights(shape), device=DEV)
    first = torch.from_numpy(np.random.default_rng(B).integers(0, vocab, size=B).astype(np.int32)).to(DEV)
    g = P.Sampling("greedy")
    a, b, ws = m.new_state(B), m.new_state(B), m.new_workspace(B)
    tok, differ, clear_all = first, [], []
    for k in range(1000):
        n0 = P.SRM.kernel_launches()
        got = m.decode_step(a, tok, g, k + 1, ws)
        assert P.SRM.kernel_launches() - n0 == 1
        want, lg = m.decode_step(b, tok, g, k + 1, ws, want_logits=True)
        top = torch.topk(lg, 2, dim=-1).values
        clear = top[:, 0] - top[:, 1] > 2.0 ** -20 * lg.abs().amax(-1)          # (two orders of addition, as above)
        differ.append(((got != want) & clear).any())
        clear_all.append(clear.float().mean())
        tok = want.clone()
    assert not torch.stack(differ).any() and torch.stack(clear_all).mean() > 0.9
    assert a.status() == 0 and b.status() == 0 and torch.equal(a.cache(), b.cache())


@pytest.mark.parametrize("B,d,vocab,mode,want_logits,inside", [
    (448, 512, 12288, "greedy", False, True), (64, 512, 12296, "greedy", False, False), (112, 512, 12296, "greedy", True, True),
    (113, 512, 12296, "greedy", True, False), (448, 512, 12288, "topk", False, True), (1, 512, 12296, "topk", False, False),
    (300, 512, 5000, "topp", False, True), (16, 512, 16392, "topp", False, True), (17, 512, 16392, "topp", True, False),
    (1, 1024, 32768, "topk", False, True), (16, 1024, 4104, "topk", True, True), (9, 1024, 32776, "topk", False, False),
    (16, 1024, 32776, "topp", False, True), (1, 1024, 32776, "greedy", True, True)])
def test_lm_head_inside_or_outside_the_layers_kernel(B, d, vocab, mode, want_logits, inside):
    """Both sides of every line between them, by the number of launches; logits against the kernel-per-operation path, tokens against the selection
    kernels run on those logits."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=2, d_model=d, vocab=vocab, n_ctx=8, dtype="bf16", seed=24)
    W = I.make_weights(shape)
    samp = {"greedy": P.Sampling("greedy"), "topk": P.Sampling("topk", 40, 0.8, seed=3, sample_idx_base=5),
            "topp": P.Sampling("topp", temperature=0.7, seed=4, sample_idx_base=6, top_p=0.9)}[mode]
    toks = torch.from_numpy(np.random.default_rng(B).integers(0, vocab, size=(3, B)).astype(np.int32)).to(DEV)
    m, ref = P.SRM(shape, W, device=DEV), P.SRM(shape, W, device=DEV, flags=P.FLAG_NO_SMALL_BATCH)
    a, b, c, ws = m.new_state(B), m.new_state(B), ref.new_state(B), ref.new_workspace(B)
    own_head = mode == "topk" and not want_logits          # (a selection of its own where the head is outside)
    for k in range(3):
        got, lg = m.decode_step(a, toks[k], samp, k + 1, ws, want_logits=True)
        n0 = P.SRM.kernel_launches()
        want = torch.empty_like(got)
        m.k_select(lg, samp, k + 1, want)
        selection, n0 = P.SRM.kernel_launches() - n0, P.SRM.kernel_launches()
        tok = m.decode_step(b, toks[k], samp, k + 1, ws, want_logits=want_logits)
        n = P.SRM.kernel_launches() - n0
        if inside:
            assert n == (1 if mode == "greedy" else 1 + selection)
        else:
            assert n == 2 + selection or (own_head and n > 2)
        assert torch.equal(got, want)
        if inside or want_logits or mode != "greedy":      # (greedy without logits outside: columns of one tile in another order of addition)
            assert torch.equal(tok[0] if want_logits else tok, got)
        lr = ref.decode_step(c, toks[k], samp, k + 1, ws, want_logits=True)[1]
        assert rel_err_rows(lg.cpu().numpy(), lr.cpu().numpy()) < 5 * 2.0 ** -9 * 2 ** 0.5          # (as above, two layers)
    assert a.status() == 0 and b.status() == 0 and torch.equal(a.cache(), b.cache())
