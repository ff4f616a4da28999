"""Kernels whose CTAs wait for one another, from two threads on streams of different priority at once (the layers kernel of
decode passes): each gives what it gives alone."""
import threading

import numpy as np
import pytest
import torch

import srm_inputs as I
from helpers import custom_shape

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B", [(256, 100), (33, 500)])
def test_two_streams_of_different_priority(B):
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=3, d_model=1024, vocab=1024, n_ctx=40, dtype="bf16", seed=31)
    W = I.make_weights(shape)
    models = [P.SRM(shape, W, device=DEV) for _ in B]
    g = P.Sampling("greedy")

    def run(i, stream, out):
        with torch.cuda.stream(stream):
            st, ws = models[i].new_state(B[i]), models[i].new_workspace(B[i], 2, prefill_samples=B[i])
            toks = torch.from_numpy(np.random.default_rng(i).integers(0, shape.vocab, size=(B[i], 2)).astype(np.int32)).to(DEV)
            models[i].prefill(st, toks, g, ws)
            gen = models[i].generate(st, 24, 1, g, ws)
            stream.synchronize()
            out[i] = (gen.clone(), st.cache(), st.status())

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
        assert both[i][2] == 0 and torch.equal(both[i][0], alone[i][0]) and torch.equal(both[i][1], alone[i][1])
