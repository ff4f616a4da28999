"""Decode passes whose layers run as one kernel, at the edges of the tile widths and row blocks of layers_mid.cuh (mixed heads with F = 4 d
of up to 448 rows at d = 512 and 112 at d = 1024 take the clusters of layers_cluster.cuh; captured steps and two streams of the kernel over the
grid are in test_gpu_decode_routes.py): logits,
tokens and cache against the kernel-per-operation path fed the same tokens (same products, sums in another order: the
bound is the one the paths with and without ranges of K are held to), a row of the batch against the oracle, equal and
per-sample positions, and the captured step."""
import numpy as np
import pytest
import torch

import srm_inputs as I
from helpers import custom_shape, oracle_for, rel_err_rows, top2_margin

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _launches(P, f):
    n0 = P.SRM.kernel_launches()
    f()
    return P.SRM.kernel_launches() - n0


@pytest.mark.parametrize("B,d,state_dtype,ragged", [(72, 512, "fp32", False), (97, 512, "fp16", True), (256, 1024, "fp16", False), (257, 1024, "fp32", True),
                                                    (512, 1024, "bf16", False), (33, 1024, "fp32", False), (130, 1536, "fp32", True),
                                                    (256, 1536, "fp16", False), (1, 1536, "fp32", False), (1000, 512, "fp32", False)])
def test_layers_in_one_kernel_agree_with_the_kernel_per_operation_path(B, d, state_dtype, ragged):
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=3, d_model=d, vocab=2048, n_ctx=24, dtype="bf16", seed=11)
    W = I.make_weights(shape)
    rng = np.random.default_rng(B)
    n = 5
    prompts_np = rng.integers(0, shape.vocab, size=(B, n)).astype(np.int32)
    lens_np = rng.integers(1, n + 1, size=B).astype(np.int32) if ragged else np.full(B, n, np.int32)
    prompts, lens = torch.from_numpy(prompts_np).to(DEV), torch.from_numpy(lens_np).to(DEV)
    g = P.Sampling("greedy")
    outs, fed = [], None
    for flags in (P.FLAG_NO_SMALL_BATCH, 0):                   # the second run consumes the first run's tokens
        m = P.SRM(shape, W, device=DEV, flags=flags, state_dtype=state_dtype)
        st, ws = m.new_state(B), m.new_workspace(B, n, prefill_samples=B)
        tok = m.prefill_ragged(st, prompts, lens, g, ws) if ragged else m.prefill(st, prompts, g, ws)
        lgs, toks = [], [tok.clone()]
        for k in range(3):
            res = []
            launches = _launches(P, lambda: res.append(m.decode_step(st, tok if fed is None else fed[k], g, k + 1, ws, want_logits=True)))
            tok, lg = res[0]
            lgs.append(lg.cpu().numpy())
            toks.append(tok.clone())
        assert (launches <= 4) == (flags == 0)                 # counters, layers and norm, LM head, selection
        assert st.status() == 0
        fed = fed if fed is not None else toks
        outs.append((np.stack(lgs), torch.stack(toks).cpu().numpy(), st.cache().cpu().numpy()))
    (lg_a, tok_a, S_a), (lg_b, tok_b, S_b) = outs
    # Sums in another order flip roundings of bf16 activations, 2^-8 of the value each. Were half of them flipped, a
    # layer would move its output by 2^-9 of its scale, three layers by 2^-9 sqrt(3); five standard deviations of that:
    tol = 5 * 2.0 ** -9 * 3 ** 0.5
    assert rel_err_rows(lg_b, lg_a) < tol and rel_err_rows(S_b, S_a) < tol
    differ = tok_a[1:] != tok_b[1:]
    assert np.all(top2_margin(lg_a)[differ] < 2e-2)
    orc = oracle_for(shape, W)
    for b in (0, B // 2, B - 1):
        lo, state = orc.forward_parallel(prompts_np[b:b + 1, :lens_np[b]])
        for k in range(3):
            lo, state = orc.decode_step(state, tok_a[k][b:b + 1], int(lens_np[b]) + k)
            assert rel_err_rows(lg_b[k][b:b + 1], lo) < 3e-2


def test_captured_step_and_passes_of_one_kernel_equal_launch_by_launch():
    """300 rows in one pass; the same steps replayed from a graph; and 300 rows as passes of 150 (rows in clusters, all three)."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=3, d_model=512, vocab=1024, n_ctx=24, dtype="bf16", seed=12)
    W = I.make_weights(shape)
    B = 300
    prompts = torch.from_numpy(np.random.default_rng(3).integers(0, shape.vocab, size=(B, 4)).astype(np.int32)).to(DEV)
    samp = P.Sampling("topk", 50, 0.8, seed=5, sample_idx_base=7)
    res = []
    for flags, chunk in ((P.FLAG_NO_GRAPH, B), (P.FLAG_GRAPH, B), (P.FLAG_NO_GRAPH, 150)):
        m = P.SRM(shape, W, device=DEV, flags=flags)
        st, ws = m.new_state(B), m.new_workspace(chunk, 4, prefill_samples=chunk)
        first = m.prefill(st, prompts, samp, ws)
        out = m.generate(st, 8, 1, samp, ws)
        assert st.status() == 0
        res.append((first.clone(), out.clone(), st.cache().clone()))
    for r in res[1:]:
        for x, y in zip(res[0], r):
            assert torch.equal(x, y)


@pytest.mark.parametrize("mixer,k,B,d,state_dtype", [("combined", 1, 12, 1024, "fp32"), ("combined", 1, 300, 512, "fp16"),
                                                     ("kernel", 1, 40, 512, "fp32"), ("kernel", 4, 257, 1024, "fp32"),
                                                     ("kernel", 5, 97, 512, "fp16"), ("kernel", 16, 130, 1024, "fp16"),
                                                     ("kernel", 13, 1000, 512, "fp32")])
def test_further_mixers_in_one_kernel_agree_with_the_kernel_per_operation_path(mixer, k, B, d, state_dtype):
    import dataclasses

    import paper_2605_08696_b200 as P
    base = custom_shape(n_layers=3, d_model=d, vocab=16384, n_ctx=24, dtype="bf16", seed=13)
    shape = dataclasses.replace(base, mixer=mixer, kernel_size=k)
    W = I.make_weights(shape)
    n = 4
    toks = torch.from_numpy(np.random.default_rng(B).integers(0, shape.vocab, size=(n + 3, B)).astype(np.int32)).to(DEV)
    g = P.Sampling("greedy")
    outs = []
    for flags in (P.FLAG_NO_SMALL_BATCH, 0):
        m = P.SRM(shape, W, device=DEV, flags=flags, state_dtype=state_dtype)
        st, ws = m.new_state(B), m.new_workspace(B, n, prefill_samples=B)
        m.prefill(st, toks[:n].t().contiguous(), g, ws)
        lgs = []
        for i in range(3):
            launches = _launches(P, lambda: lgs.append(m.decode_step(st, toks[n + i], g, i + 1, ws, want_logits=True)[1].cpu().numpy()))
        assert (launches <= 4) == (flags == 0) and st.status() == 0
        outs.append((np.stack(lgs), st.cache().cpu().numpy()))
    tol = 5 * 2.0 ** -9 * 3 ** 0.5                             # as above
    assert rel_err_rows(outs[1][0], outs[0][0]) < tol and rel_err_rows(outs[1][1], outs[0][1]) < tol
    orc = oracle_for(shape, W)
    for b in (0, B - 1):
        lo, state = orc.forward_parallel(toks[:n, b:b + 1].t().cpu().numpy())
        for i in range(3):
            lo, state = orc.decode_step(state, toks[n + i, b:b + 1].cpu().numpy(), n + i)
            assert rel_err_rows(outs[1][0][i][b:b + 1], lo) < 3e-2


@pytest.mark.parametrize("B,d,mult,heads,layers,state_dtype,ragged", [
    (1, 320, 4, 4, 3, "fp32", False), (64, 320, 4, 8, 3, "bf16", True), (33, 448, 4, 4, 3, "fp16", False),
    (8, 512, 3, 4, 3, "fp32", False), (3, 512, 5, 8, 3, "fp32", True), (64, 512, 12, 4, 3, "fp16", False),
    (17, 640, 2, 4, 3, "fp32", False), (64, 768, 8, 4, 3, "fp32", True), (9, 832, 4, 4, 1, "fp32", False),
    (40, 832, 5, 8, 3, "fp16", False), (1, 960, 6, 4, 3, "fp32", True), (63, 960, 6, 6, 3, "bf16", False), (64, 960, 4, 4, 2, "fp32", False),
    (100, 512, 4, 8, 1, "fp32", False), (75, 512, 4, 8, 3, "bf16", True), (130, 1536, 4, 8, 1, "fp16", True)])
def test_models_of_any_width_and_head_count(B, d, mult, heads, layers, state_dtype, ragged):
    """Widths and hidden widths the single-kernel step is not built for, up to 64 rows: rows that do not fill the threads,
    k-blocks that do not fill a stage (d = 64 x odd), last column tiles partly filled (F = 5760 in tiles of 128), ranges of K of
    unequal length (F = 3328, 5760). And heads that are not whole multiples of 128 channels (the partial products then lie in
    the logits area); models of a single layer."""
    import dataclasses

    import paper_2605_08696_b200 as P
    base = custom_shape(n_layers=layers, d_model=d, vocab=16384 if d == 1536 else 4096, n_ctx=24, dtype="bf16", seed=17)
    shape = dataclasses.replace(base, ffn_mult=mult, n_heads=heads)
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
        m.prefill_ragged(st, prompts, lens, g, ws) if ragged else m.prefill(st, prompts, g, ws)
        lgs = []
        for k in range(3):
            launches = _launches(P, lambda: lgs.append(m.decode_step(st, fed[k], g, k + 1, ws, want_logits=True)[1].cpu().numpy()))
        assert (launches <= 4) == (flags == 0)                 # counters, layers and norm, LM head, selection
        assert st.status() == 0
        outs.append((np.stack(lgs), st.cache().cpu().float().numpy()))
    (lg_a, S_a), (lg_b, S_b) = outs
    tol = 5 * 2.0 ** -9 * layers ** 0.5                        # as above
    assert rel_err_rows(lg_b, lg_a) < tol and rel_err_rows(S_b, S_a) < tol
    orc = oracle_for(shape, W)
    for b in (0, B - 1):
        lo, state = orc.forward_parallel(prompts_np[b:b + 1, :lens_np[b]])
        for k in range(3):
            lo, state = orc.decode_step(state, fed[k, b:b + 1].cpu().numpy(), int(lens_np[b]) + k)
            assert rel_err_rows(lg_b[k][b:b + 1], lo) < 3e-2
