"""Prefill through the chunk kernel (csrc/prefill_chunk.cuh: a chunk of 16 positions per CTA, end states handed on
through scratch memory) at the edges of its chunks, against the fp64 oracle's parallel form (fp32 model: plain FMA
everywhere, so the comparison is at the fp32 tolerance)."""
import numpy as np
import pytest
import torch

import srm_inputs as I
from helpers import oracle_for, rel_err_rows
from parity import DEV, TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,B", [(512, 1, 3), (512, 16, 2), (512, 17, 5), (1024, 33, 2), (1024, 15, 40), (1536, 64, 2), (2048, 49, 1),
                                   (512, 700, 1)])
def test_prefill_in_chunks_matches_the_oracle(d, n, B):
    import paper_2605_08696_b200 as P
    shape = I.SRMShape(n_layers=2, d_model=d, vocab=64, n_ctx=max(n, 16) + 2, ffn_mult=1 if d == 2048 else 2, dtype="fp32", seed=d + n)
    W = I.make_weights(shape)
    orc = oracle_for(shape, W)
    model = P.SRM(shape, W, device=DEV)
    toks = I.uniform_prompts(B, n, shape.vocab, seed=n)
    dev = torch.from_numpy(toks).to(DEV)
    g = P.Sampling("greedy")
    ws = model.new_workspace(B, n, prefill_samples=B)
    st = model.new_state(B)
    _, lg = model.prefill(st, dev, g, ws, want_logits=True)
    few = np.unique(np.linspace(0, B - 1, min(B, 4)).astype(int))
    lo, so = orc.forward_parallel(toks[few])
    assert rel_err_rows(lg.cpu().numpy()[few], lo[:, n - 1]) < TOL["fp32"]
    cache = st.cache().cpu().numpy()
    for l in range(shape.n_layers):
        assert rel_err_rows(cache[l][few], so[l]) < TOL["fp32"]
    # prompts of different lengths: every sample as if it were alone (chunks past its length only clear their rows)
    lens = np.maximum(1, n - np.arange(B) % max(1, n)).astype(np.int32)
    s2 = model.new_state(B)
    model.prefill_ragged(s2, dev, torch.from_numpy(lens).to(DEV), g, ws)
    c2 = s2.cache().cpu().numpy()
    for b in few:
        _, sb = orc.forward_parallel(toks[b:b + 1, :lens[b]])
        for l in range(shape.n_layers):
            assert rel_err_rows(c2[l][b:b + 1], sb[l]) < TOL["fp32"]
    assert st.status() == 0 and s2.status() == 0


@pytest.mark.parametrize("mixer,k,d,n,B", [("combined", 1, 512, 40, 3), ("combined", 1, 1024, 16, 2), ("kernel", 1, 512, 17, 3),
                                           ("kernel", 3, 1024, 49, 2), ("kernel", 4, 512, 32, 2), ("kernel", 7, 1024, 18, 3),
                                           ("kernel", 16, 1024, 33, 2), ("kernel", 16, 512, 1, 2)])
def test_prefill_in_chunks_of_the_further_mixers_matches_the_oracle(mixer, k, d, n, B):
    """bf16 models. The cache of layer 0 sees only fp32 arithmetic (embedding, LN1, recurrence): fp32 tolerance. Layer 1
    and the logits come through the bf16 feed-forward: bf16 tolerance; a wrong y (a wrapped channel, a shift) moves
    them by far more."""
    import paper_2605_08696_b200 as P
    shape = I.SRMShape(n_layers=2, d_model=d, vocab=64, n_ctx=64, dtype="bf16", seed=d + n + k, mixer=mixer, kernel_size=k)
    W = I.make_weights(shape, alpha_std=0.3)
    model = P.SRM(shape, W, device=DEV)
    toks = I.uniform_prompts(B, n, shape.vocab, seed=n)
    st = model.new_state(B)
    ws = model.new_workspace(B, n, prefill_samples=B)
    _, lg = model.prefill(st, torch.from_numpy(toks).to(DEV), P.Sampling("greedy"), ws, want_logits=True)
    lo, so = oracle_for(shape, W).forward_parallel(toks)
    cache = st.cache().cpu().numpy()
    assert rel_err_rows(cache[0], so[0]) < TOL["fp32"]
    assert rel_err_rows(cache[1], so[1]) < TOL["bf16"]
    assert rel_err_rows(lg.cpu().numpy(), lo[:, n - 1]) < TOL["bf16"]
    assert st.status() == 0
