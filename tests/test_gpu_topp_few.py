"""Top-p rows with a small nucleus (select_topp_few_kernel: the row in registers, the nucleus ranked among the few tokens
near the maximum) against the oracle's sampler, at the edges: vocabularies that fill the registers and one that does not fit
(the general kernel alone), ties at the nucleus edge, as many near tokens as fit and one more, a nucleus that reaches past
them, rows handed to the general kernel. Both kernels give the same tokens, so which of them settled a row shows in the time."""
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


def test_rows_with_few_near_tokens_are_settled_by_the_first_kernel():
    """Rows handed on are walked by one block per SM, three to five times the time per row (3000 rows of 32000: 192 us when the
    first kernel settles all of them, 939 through the general one): 256 near tokens must be settled in the first pass, 257 and
    flat rows must not, in a vocabulary that fits the registers; in one that does not, no row is."""
    import paper_2605_08696_b200 as P
    R = 2000
    samp = P.Sampling("topp", temperature=0.7, seed=17, sample_idx_base=50, top_p=0.9)

    def us(V, near):
        shape = custom_shape(n_layers=1, d_model=64, vocab=V, n_ctx=8, dtype="fp32", seed=3)
        model = P.SRM(shape, I.make_weights(shape), device=DEV)
        lg = torch.randn(R, V, generator=torch.Generator(device=DEV).manual_seed(V), device=DEV)
        if near:
            lg[:, 7:7 + near] = 20.0
        tok, status = torch.zeros(R, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            model.k_select(lg, samp, 0, tok, status)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        assert int(status.item()) == 0
        return sorted(times[2:])[2]

    few, full, over, flat = us(32000, 4), us(32000, 256), us(32000, 257), us(32000, 0)
    assert max(few, full) < 0.6 * min(over, flat), (few, full, over, flat)
    edge, past = us(32768, 4), us(32776, 4)
    assert edge < 0.6 * past, (edge, past)
