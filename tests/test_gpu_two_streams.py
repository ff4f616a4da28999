"""Kernels whose CTAs wait for one another, from two threads on streams of different priority at once (the layers kernel of
decode passes, the feed-forward kernel of prefills and of larger decode passes): each gives what it gives alone. (100 and 33 rows run in
clusters that wait for nobody; two kernels over the grid on both sides are in test_gpu_decode_routes.py.)"""
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


@pytest.mark.parametrize("sides,ffn", [([(256, 12, 4), (250, 12, 4)], (True, True)),          # two prefills of 3000 rows
                                       ([(256, 12, 4), (256, 2, 24)], (True, False)),         # a prefill beside steps of the layers kernel
                                       ([(256, 2, 24), (2304, 2, 8)], (False, True)),         # these beside larger decode passes
                                       ([(2304, 2, 8), (1500, 12, 4)], (True, True))])        # these beside a prefill in two slabs
def test_feed_forward_kernels_on_two_streams(sides, ffn):
    """sides: (samples, prompt length, steps); ffn: whether the side runs the feed-forward kernel."""
    import paper_2605_08696_b200 as P
    shape = custom_shape(n_layers=3, d_model=1024, vocab=1024, n_ctx=40, dtype="bf16", seed=31)
    W = I.make_weights(shape)
    models = [P.SRM(shape, W, device=DEV) for _ in sides]
    g = P.Sampling("greedy")

    def run(i, stream, out):
        B, n, steps = sides[i]
        with torch.cuda.stream(stream):
            st, ws = models[i].new_state(B), models[i].new_workspace(B, n, prefill_samples=B)
            toks = torch.from_numpy(np.random.default_rng(i).integers(0, shape.vocab, size=(B, n)).astype(np.int32)).to(DEV)
            res = []
            for _ in range(3):
                st.reset()
                res += [models[i].prefill(st, toks, g, ws).clone(), models[i].generate(st, steps, 1, g, ws).clone(), st.cache()]
            stream.synchronize()
            out[i] = (res, st.status())

    alone, both = {}, {}
    for i in range(2):
        models[i].profile(True)
        run(i, torch.cuda.Stream(), alone)
        assert (models[i].profile_read()["ffn"][0] > 0) == ffn[i]
        models[i].profile(False)
    streams = [torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)]
    threads = [threading.Thread(target=run, args=(i, streams[i], both)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(2):
        assert both[i][1] == 0 and all(torch.equal(x, y) for x, y in zip(both[i][0], alone[i][0]))
