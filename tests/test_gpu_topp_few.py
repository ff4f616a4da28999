"""Top-p rows with a small nucleus (select_topp_few_kernel: the row in registers, the nucleus ranked among the few tokens
near the maximum) against the oracle's sampler, at the edges: vocabularies that fill the registers, ties at the nucleus
edge, as many near tokens as fit and one more, a nucleus that reaches past them, rows handed to the general kernel."""
import numpy as np
import pytest
import torch

from helpers import custom_shape, topp_is_strict
import srm_inputs as I

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("V", [8, 2048, 8000, 32000, 32768, 32776])
def test_small_nucleus_rows_equal_the_oracle(V):
    import paper_2605_08696_b200 as P
    from oracle import srm_oracle as O
    shape = custom_shape(n_layers=1, d_model=64, vocab=V, n_ctx=8, dtype="fp32", seed=3)
    model = P.SRM(shape, I.make_weights(shape), device=DEV)
    rng = np.random.default_rng(V)
    R = 40
    lg = rng.normal(0, 1, size=(R, V)).astype(np.float32)
    for r in range(R):
        k = [1, 2, 4, 7][r % 4]
        ids = rng.choice(V, size=min(k, V - 1), replace=False)
        lg[r, ids] = 14.0 + rng.normal(0, 1, size=len(ids)).astype(np.float32)
        if r % 5 == 0:
            lg[r, ids] = 15.0                                     # equal: the lowest ids are in
    if V >= 2048:
        lg[1, rng.choice(V, size=256, replace=False)] = 20.0      # exactly as many near tokens as fit, all ties
        lg[2, rng.choice(V, size=257, replace=False)] = 20.0      # one more: the general kernel
        lg[3] = rng.normal(0, 0.1, size=V)                        # flat: the general kernel
        lg[6, 0] = 7.5                                            # the nucleus may reach past the near tokens
    T, p = 0.7, 0.9
    samp = P.Sampling("topp", temperature=T, seed=17, sample_idx_base=50, top_p=p)
    dev = torch.from_numpy(lg).to(DEV)
    checked = 0
    for step in range(4):
        tok = torch.full((R,), -7, dtype=torch.int32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        model.k_select(dev, samp, step, tok, status)
        got = tok.cpu().numpy()
        want, det = O.select_topp(lg, np.float32(p), T, 17, 50 + np.arange(R), step, return_detail=True)
        assert int(status.item()) == 0
        for r in range(R):
            if topp_is_strict(lg[r], float(np.float32(p)), T, det[r]):
                assert got[r] == want[r], (step, r)
                checked += 1
    assert checked > 0.9 * 4 * R
