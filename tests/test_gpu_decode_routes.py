"""Every kernel that takes a decode pass whole, on sizes that are its own (the route is asked for, not inferred): the single-kernel
step at the widths, hidden widths and head counts that the cluster kernels leave to it; the layers kernel over the grid, replayed and on two
streams; the kernel with its weights split between clusters under generate, captured, sampled and in passes."""
import dataclasses
import threading

import numpy as np
import pytest
import torch

import srm_inputs as I
from helpers import custom_shape, oracle_for, rel_err_rows, top2_margin, topp_is_strict

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _shape(d, vocab=2048, layers=3, n_ctx=40, mult=4, heads=4, seed=41):
    return dataclasses.replace(custom_shape(n_layers=layers, d_model=d, vocab=vocab, n_ctx=n_ctx, dtype="bf16", seed=seed), ffn_mult=mult, n_heads=heads)


def _tokens(seed, vocab, *size):
    return torch.from_numpy(np.random.default_rng(seed).integers(0, vocab, size=size).astype(np.int32)).to(DEV)


@pytest.mark.parametrize("d,mult,heads,B,route", [
    (512, 4, 4, 1, "clusters"), (512, 4, 4, 64, "clusters"), (512, 4, 4, 72, "clusters"), (512, 4, 4, 448, "clusters"), (512, 4, 4, 449, "layers"),
    (512, 4, 8, 7, "clusters"), (512, 2, 4, 64, "step"), (512, 4, 4, 1001, "layers"), (512, 4, 4, 1200, "kernels"),
    (1024, 4, 4, 1, "split"), (1024, 4, 4, 16, "split"), (1024, 4, 4, 17, "clusters"), (1024, 4, 4, 112, "clusters"), (1024, 4, 4, 113, "layers"),
    (1024, 4, 8, 16, "split"), (1024, 4, 2, 17, "clusters"), (1024, 3, 4, 16, "step"), (1024, 4, 4, 512, "layers"), (1024, 4, 4, 513, "kernels"),
    (256, 4, 4, 64, "step"), (768, 4, 4, 48, "step"), (768, 4, 4, 65, "kernels"), (320, 4, 4, 20, "layers"), (1536, 4, 4, 1, "layers"), (1536, 4, 4, 256, "layers")])
def test_route_of_a_pass(d, mult, heads, B, route):
    import paper_2605_08696_b200 as P
    shape = _shape(d, vocab=16384, layers=1, mult=mult, heads=heads)
    W = I.make_weights(shape)
    m = P.SRM(shape, W, device=DEV)
    assert m.decode_route(B, m.new_workspace(B)) == route
    off = P.SRM(shape, W, device=DEV, flags=P.FLAG_NO_SMALL_BATCH)
    assert off.decode_route(B, off.new_workspace(B)) == "kernels"


@pytest.mark.parametrize("d,mult,heads,B,state_dtype,ragged", [
    (256, 4, 4, 64, "fp32", False), (512, 2, 4, 48, "fp32", True), (512, 6, 4, 1, "fp16", False), (768, 4, 4, 33, "bf16", False), (768, 4, 6, 3, "fp32", True),
    (1024, 3, 4, 16, "fp16", False), (1024, 2, 4, 1, "fp32", False), (1024, 3, 8, 7, "bf16", True)])
def test_single_kernel_step_of_the_models_it_serves(d, mult, heads, B, state_dtype, ragged):
    """Against the kernel-per-operation path fed the same tokens and, by rows, the oracle; generated from a graph and launch by launch."""
    import paper_2605_08696_b200 as P
    shape = _shape(d, mult=mult, heads=heads)
    W = I.make_weights(shape)
    n, g = 5, P.Sampling("greedy")
    prompts_np = np.random.default_rng(B).integers(0, shape.vocab, size=(B, n)).astype(np.int32)
    lens_np = np.random.default_rng(B + 1).integers(1, n + 1, size=B).astype(np.int32) if ragged else np.full(B, n, np.int32)
    prompts, lens, fed = torch.from_numpy(prompts_np).to(DEV), torch.from_numpy(lens_np).to(DEV), _tokens(3, shape.vocab, 3, B)

    def prefilled(m, ws):
        st = m.new_state(B)
        m.prefill_ragged(st, prompts, lens, g, ws) if ragged else m.prefill(st, prompts, g, ws)
        return st

    outs = []
    for flags in (P.FLAG_NO_SMALL_BATCH, 0):
        m = P.SRM(shape, W, device=DEV, flags=flags, state_dtype=state_dtype)
        ws = m.new_workspace(B, n, prefill_samples=B)
        assert m.decode_route(B, ws) == ("kernels" if flags else "step")
        st = prefilled(m, ws)
        lgs = [m.decode_step(st, f, g, k + 1, ws, want_logits=True)[1].cpu().numpy() for k, f in enumerate(fed)]
        assert st.status() == 0
        outs.append((np.stack(lgs), st.cache().cpu().float().numpy()))
    tol = 5 * 2.0 ** -9 * 3 ** 0.5                 # flipped roundings of bf16 activations over three layers (test_gpu_layers_mid.py)
    assert rel_err_rows(outs[1][0], outs[0][0]) < tol and rel_err_rows(outs[1][1], outs[0][1]) < tol
    orc = oracle_for(shape, W)
    for b in {0, B // 2, B - 1}:
        lo, state = orc.forward_parallel(prompts_np[b:b + 1, :lens_np[b]])
        for k in range(3):
            lo, state = orc.decode_step(state, fed[k, b:b + 1].cpu().numpy(), int(lens_np[b]) + k)
            assert rel_err_rows(outs[1][0][k][b:b + 1], lo) < 3e-2
    gen = []
    for flags in (P.FLAG_NO_GRAPH, P.FLAG_GRAPH):
        m = P.SRM(shape, W, device=DEV, flags=flags, state_dtype=state_dtype)
        ws = m.new_workspace(B, n, prefill_samples=B)
        st = prefilled(m, ws)
        gen.append((m.generate(st, 8, 1, g, ws).clone(), st.cache().clone()))
        assert st.status() == 0
    assert torch.equal(gen[0][0], gen[1][0]) and torch.equal(gen[0][1], gen[1][1])


def _generated(P, shape, W, B, flags, samp, route, chunk=None, steps=12):
    m = P.SRM(shape, W, device=DEV, flags=flags)
    st, ws = m.new_state(B), m.new_workspace(chunk or B, 4, prefill_samples=chunk or B)
    assert m.decode_route(chunk or B, ws) == route
    first = m.prefill(st, _tokens(9, shape.vocab, B, 4), samp, ws).clone()
    out = m.generate(st, steps, 1, samp, ws).clone()
    assert st.status() == 0
    return first, out, st.cache().clone()


@pytest.mark.parametrize("B,d,route", [(500, 512, "layers"), (300, 1024, "layers"), (1, 1024, "split"), (16, 1024, "split"), (27, 1024, "clusters"),
                                       (300, 512, "clusters")])
@pytest.mark.parametrize("mode", ["greedy", "topk", "topp"])
def test_generate_from_a_graph_equals_launch_by_launch(B, d, route, mode):
    """... and steps called one by one."""
    import paper_2605_08696_b200 as P
    shape = _shape(d)
    W = I.make_weights(shape)
    samp = {"greedy": P.Sampling("greedy"), "topk": P.Sampling("topk", 50, 0.8, seed=5, sample_idx_base=7),
            "topp": P.Sampling("topp", temperature=0.7, seed=6, sample_idx_base=3, top_p=0.9)}[mode]
    a, b = (_generated(P, shape, W, B, f, samp, route) for f in (P.FLAG_NO_GRAPH, P.FLAG_GRAPH))
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    m = P.SRM(shape, W, device=DEV)
    st, ws = m.new_state(B), m.new_workspace(B, 4, prefill_samples=B)
    tok = m.prefill(st, _tokens(9, shape.vocab, B, 4), samp, ws)
    for k in range(12):
        tok = m.decode_step(st, tok, samp, k + 1, ws).clone()
        assert torch.equal(tok, a[1][:, k])
    assert torch.equal(st.cache(), a[2])


def test_a_batch_in_passes_of_the_split_kernel_equals_batches_of_their_size():
    import paper_2605_08696_b200 as P
    shape = _shape(1024)
    W = I.make_weights(shape)
    m = P.SRM(shape, W, device=DEV)
    toks, g = _tokens(11, shape.vocab, 5, 40), P.Sampling("greedy")
    whole, ws = m.new_state(40), m.new_workspace(16)
    parts = [(b, m.new_state(min(16, 40 - b))) for b in (0, 16, 32)]
    assert m.decode_route(40, ws) == "split"
    for k, t in enumerate(toks):
        got, lg = m.decode_step(whole, t, g, k + 1, ws, want_logits=True)
        for b, st in parts:
            want, lw = m.decode_step(st, t[b:b + st.B].contiguous(), g, k + 1, ws, want_logits=True)
            assert torch.equal(got[b:b + st.B], want) and torch.equal(lg[b:b + st.B], lw)
    assert whole.status() == 0
    for b, st in parts:
        assert torch.equal(whole.cache()[:, b:b + st.B], st.cache())


@pytest.mark.parametrize("B", [1, 16])
@pytest.mark.parametrize("mode", ["topk", "topp"])
def test_sampling_after_the_split_kernel(B, mode):
    """The oracle's sampler run on the logits of a step picks the device's token (CDF edges excepted); without logits, the same token."""
    import paper_2605_08696_b200 as P
    from oracle import srm_oracle as O
    shape = _shape(1024, vocab=4096)
    m = P.SRM(shape, I.make_weights(shape), device=DEV)
    samp = P.Sampling("topk", 50, 0.8, seed=21, sample_idx_base=300) if mode == "topk" else P.Sampling("topp", temperature=0.7, seed=21, sample_idx_base=300, top_p=0.9)
    a, b, ws = m.new_state(B), m.new_state(B), m.new_workspace(B)
    assert m.decode_route(B, ws) == "split"
    tok, checked, steps = _tokens(B, shape.vocab, B), 0, 24 if B == 1 else 4
    for k in range(1, steps + 1):
        got, lg = m.decode_step(a, tok, samp, k, ws, want_logits=True)
        assert torch.equal(m.decode_step(b, tok, samp, k, ws), got)
        lg_np, t = lg.cpu().numpy(), got.cpu().numpy()
        if mode == "topk":
            want, det = O.select_topk(lg_np, 50, 0.8, 21, 300 + np.arange(B), k, return_detail=True)
        else:
            want, det = O.select_topp(lg_np, np.float32(0.9), 0.7, 21, 300 + np.arange(B), k, return_detail=True)
        for r in range(B):
            if mode == "topk":
                c, thr = det[r]["cdf"], det[r]["thr"]
                strict = np.min(np.abs(c - thr)) / c[-1] > 1e-5          # (fp32 weights of at most 50 tokens against fp64)
            else:
                strict = topp_is_strict(lg_np[r], float(np.float32(0.9)), 0.7, det[r])
            if strict:
                assert want[r] == t[r]
                checked += 1
        tok = got.clone()
    assert checked > 0.9 * steps * B and a.status() == 0 and b.status() == 0


@pytest.mark.parametrize("B,routes", [((256, 130), ("layers", "layers")), ((120, 500), ("layers", "layers")), ((16, 256), ("split", "layers")),
                                      ((1, 16), ("split", "split")), ((16, 100), ("split", "clusters")), ((100, 300), ("clusters", "layers"))])
def test_two_streams_of_different_priority(B, routes):
    """Two threads' generations at once, kernels whose CTAs wait for one another on both sides: each gives what it gives alone."""
    import paper_2605_08696_b200 as P
    shape = _shape(1024, vocab=1024)
    W = I.make_weights(shape)
    models = [P.SRM(shape, W, device=DEV) for _ in B]
    g = P.Sampling("greedy")

    def run(i, stream, out):
        with torch.cuda.stream(stream):
            st, ws = models[i].new_state(B[i]), models[i].new_workspace(B[i], 2, prefill_samples=B[i])
            assert models[i].decode_route(B[i], ws) == routes[i]
            res = []
            for _ in range(3):
                st.reset()
                models[i].prefill(st, _tokens(i, shape.vocab, B[i], 2), g, ws)
                res += [models[i].generate(st, 30, 1, g, ws).clone(), st.cache().clone()]
            stream.synchronize()
            out[i] = (res, st.status())

    alone, both = {}, {}
    for i in range(2):
        run(i, torch.cuda.Stream(), alone)
    streams = [torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)]
    threads = [threading.Thread(target=run, args=(i, streams[i], both)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(2):
        assert both[i][1] == 0 and all(torch.equal(x, y) for x, y in zip(both[i][0], alone[i][0]))


@pytest.mark.parametrize("B,d", [(1, 512), (40, 512), (300, 512), (1, 1024), (9, 1024), (27, 1024)])
def test_status_of_a_step_that_selects_in_the_layers_kernel(B, d):
    """A token id outside the vocabulary is clamped and reported; a row whose cache is not finite is reported, gets token 0 and touches no
    other row."""
    import paper_2605_08696_b200 as P
    shape = _shape(d)
    m = P.SRM(shape, I.make_weights(shape), device=DEV)
    g, tok = P.Sampling("greedy"), _tokens(B, shape.vocab, B)
    ws = m.new_workspace(B)

    def step(t, spoil=None):
        st = m.new_state(B)
        if spoil is not None:
            st.layer(0)[spoil] = float("nan")
        return m.decode_step(st, t, g, 1, ws).clone(), st

    low, high = tok.clone(), tok.clone()
    low[0], high[B - 1] = -5, shape.vocab + 7
    for bad, row, good in ((low, 0, 0), (high, B - 1, shape.vocab - 1)):
        clamped = bad.clone()
        clamped[row] = good
        (got, st), (want, ref) = step(bad), step(clamped)
        assert st.status() == 1 and ref.status() == 0 and torch.equal(got, want) and torch.equal(st.cache(), ref.cache())
    clean, _ = step(tok)
    for row in {0, B // 2, B - 1}:
        got, st = step(tok, row)
        assert st.status() == 4 and got[row].item() == 0
        others = [r for r in range(B) if r != row]
        assert torch.equal(got[others], clean[others]) and bool(st.cache()[:, others].isfinite().all())


@pytest.mark.parametrize("B,vocab,layers,logits,launches", [(32, 65544, 1, True, 1), (32, 65544, 1, False, 3), (17, 65536, 1, True, 3), (33, 65544, 1, True, 3),
                                                            (20, 73736, 9, True, 1), (20, 73728, 9, True, 3)])
def test_logits_of_a_large_vocabulary_after_few_layers(B, vocab, layers, logits, launches):
    """17 to 32 rows at d = 1024: the single-kernel step, LM head included, where logits are wanted and the vocabulary is large for the number of
    layers; the same step on kernels per operation."""
    import paper_2605_08696_b200 as P
    shape = _shape(1024, vocab=vocab, layers=layers, n_ctx=8)
    W = I.make_weights(shape)
    toks, g = _tokens(B, vocab, 2, B), P.Sampling("greedy")
    m = P.SRM(shape, W, device=DEV)
    st, ws = m.new_state(B), m.new_workspace(B)
    n0, out = P.SRM.kernel_launches(), None
    for k in range(2):
        out = m.decode_step(st, toks[k], g, k + 1, ws, want_logits=logits)
    assert P.SRM.kernel_launches() - n0 == 2 * launches and st.status() == 0
    ref = P.SRM(shape, W, device=DEV, flags=P.FLAG_NO_SMALL_BATCH)
    sr = ref.new_state(B)
    for k in range(2):
        _, lr = ref.decode_step(sr, toks[k], g, k + 1, ws, want_logits=True)
    tol = 5 * 2.0 ** -9 * layers ** 0.5                      # (as above)
    assert rel_err_rows(st.cache().cpu().numpy(), sr.cache().cpu().numpy()) < tol
    if logits:
        assert rel_err_rows(out[1].cpu().numpy(), lr.cpu().numpy()) < tol
