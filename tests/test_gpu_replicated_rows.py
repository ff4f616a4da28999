"""The cache of a prompt copied to its replicas, around the 32 replicas and 128 vectors of 16 bytes that a block copies: bit for
bit what a prefill of the replicated prompts leaves."""
import numpy as np
import pytest
import torch

import srm_inputs as I
from helpers import custom_shape

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,state_dtype,prompts,replicas", [(64, "fp16", 3, 31), (512, "fp32", 1, 33), (512, "fp32", 2, 32),
                                                            (1024, "fp16", 5, 2), (1536, "fp32", 2, 70)])
def test_replicas_hold_the_cache_of_their_prompt(d, state_dtype, prompts, replicas):
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=2, d_model=d, vocab=512, n_ctx=24, dtype="bf16" if d > 64 else "fp32", seed=21)
    model = P.SRM(shape, I.make_weights(shape), device=DEV, state_dtype=state_dtype)
    base = torch.from_numpy(np.random.default_rng(d).integers(0, shape.vocab, size=(prompts, 7)).astype(np.int32)).to(DEV)
    B = prompts * replicas
    g = P.Sampling("greedy")
    ws = model.new_workspace(B, 7, prefill_samples=B)
    a, b = model.new_state(B), model.new_state(B)
    ta = model.prefill_replicated(a, base, replicas, g, ws)
    tb = model.prefill(b, base.repeat_interleave(replicas, dim=0).contiguous(), g, ws)
    assert torch.equal(a.cache(), b.cache()) and torch.equal(ta, tb)
    assert a.status() == 0 and b.status() == 0
