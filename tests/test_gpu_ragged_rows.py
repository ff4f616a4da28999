"""Prompts of different lengths are stored one after the other for the projections of a prefill pass: the cache and the
logits of every prompt must be those of the same prompt in a pass of prompts of its own length, bit for bit (a row's
arithmetic does not depend on where the row is stored)."""
import numpy as np
import pytest
import torch

import srm_inputs as I

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("lengths,n_max", [
    ([1, 1, 1], 200),                               # three rows in all, one block of 600
    ([200, 55, 1], 200),                            # 256 rows: exactly one row block
    ([200, 56, 1], 200),                            # one row more
    ([200, 200, 200], 200),                         # nothing to pack
    ([1] * 89 + [200], 200),                        # more than one slab of rows, the second empty
    ([200] * 82 + [1] * 8, 200),                    # ... the second nearly empty
    ([3, 24] * 300, 24),                            # many prompts: a CTA per prompt
])
def test_packed_rows_give_what_each_prompt_gives_alone(lengths, n_max):
    import paper_2605_08696_b200 as P
    shape = I.CONFIGS["small"]
    model = P.SRM(shape, I.make_weights(shape), device=DEV)
    B = len(lengths)
    toks = I.uniform_prompts(B, n_max, shape.vocab, seed=11)
    g = P.Sampling("greedy")
    st = model.new_state(B)
    ws = model.new_workspace(B, n_max, prefill_samples=B)
    lens = torch.tensor(lengths, dtype=torch.int32, device=DEV)
    tok, lg = model.prefill_ragged(st, torch.from_numpy(toks).to(DEV), lens, g, ws, want_logits=True)
    assert st.status() == 0
    cache = st.cache()
    for n in sorted(set(lengths)):
        rows = [b for b in range(B) if lengths[b] == n]
        # as many prompts per pass as in the batch: the same mixer kernel
        batch = np.resize(np.asarray(rows), B)
        one = model.new_state(B)
        t1, l1 = model.prefill(one, torch.from_numpy(np.ascontiguousarray(toks[batch, :n])).to(DEV), g, ws, want_logits=True)
        idx = torch.tensor(batch, device=DEV)
        assert torch.equal(tok[idx], t1) and torch.equal(lg[idx], l1)
        assert torch.equal(cache[:, idx], one.cache())
