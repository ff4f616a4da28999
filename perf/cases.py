"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one pass through the public calls of `paper_2605_08696_b200` (`SRM.decode_step`, `generate`, `prefill`,
`prefill_ragged`, `prefill_replicated`) on one of the repository's model configurations ("small", "mid" and "rl" of
`srm_inputs.py`), from a single interactive sample to a whole rollout batch. The weights are random like those of
`srm_inputs.make_weights`, with one addition: embeddings dominate the residual stream and every LM-head row also holds
a part of the embeddings of a few predecessor tokens, so that, as in a trained model, a handful of tokens carry the
probability mass and a decision is not a tie of thousands of equal logits that any rounding flips.
"""
import functools
import math

import torch

import paper_2605_08696_b200 as srm

MODELS = {
    "small": dict(n_layers=8, d_model=512, n_heads=4, ffn_mult=4, vocab=8000, n_ctx=512, dtype="bf16", ln_eps=1e-5),
    "mid": dict(n_layers=16, d_model=1024, n_heads=4, ffn_mult=4, vocab=32000, n_ctx=1024, dtype="bf16", ln_eps=1e-5),
    "rl": dict(n_layers=24, d_model=1536, n_heads=4, ffn_mult=4, vocab=32000, n_ctx=1024, dtype="bf16", ln_eps=1e-5),
}
# Logits of the four successors of a token, and the share of a row's embedding that is left after all layers (which
# the head has to make up for): greedy models are confident, the sampled one leaves mass to several tokens.
SUCCESSORS = {"small": (18.0, 11.0, 10.0, 9.0), "mid": (18.0, 11.0, 10.0, 9.0), "rl": (14.0, 12.0, 11.0, 10.0)}
KEPT = {"small": 0.98, "mid": 0.88, "rl": 0.70}
EMBED_STD = 4.0
L2_BYTES = 100e6      # weights larger than this come from HBM again in every step

DEFAULTS = dict(do="generate", model="mid", mixer="mixed", k=1, cache="fp32", batch=1, prompt=1, steps=0, prompts=0,
                select="greedy", top_k=50, top_p=0.9, temperature=1.0, logits=False)


def _case(**kw):
    return {**DEFAULTS, **kw}


def listed():
    return [
        # one interactive sample, one token: nothing but latency
        _case(name="token_1", do="decode", batch=1, prompt=300),
        # a handful of conversations on the half-precision cache
        _case(name="chat_27", batch=27, prompt=411, steps=24, cache="fp16"),
        # the small configuration at its own batch
        _case(name="small_256", model="small", batch=256, prompt=128, steps=24),
        # a mid-sized serving batch, not a multiple of any tile
        _case(name="serve_500", batch=500, prompt=256, steps=8),
        # the throughput benchmark: 4096 samples, greedy
        _case(name="throughput_4096", batch=4096, prompt=256, steps=4),
        # a step of the rollout workload: 16384 samples, top-k sampling
        _case(name="rollout_topk_16384", do="decode", model="rl", batch=16384, prompt=200, select="topk", temperature=0.8),
        # a step of rollouts with nucleus sampling, for one question's samples
        _case(name="rollout_topp_3000", do="decode", model="rl", batch=3000, prompt=200, select="topp", temperature=0.7),
        # time to the first token of one long prompt
        _case(name="prompt_777", do="prefill", batch=1, prompt=777),
        # prefill of the throughput benchmark
        _case(name="prompts_2048x256", do="prefill", batch=2048, prompt=256),
        # a serving batch of prompts of different lengths, and its first generated tokens
        _case(name="ragged_45", do="ragged", batch=45, prompt=301, steps=4, logits=True),
        # the rollout workload's prompts: 16 questions, 1024 samples each
        _case(name="questions_16x1024", do="replicated", model="rl", batch=16384, prompts=16, prompt=200, select="topk",
              temperature=0.8),
        # the further token mixers: kernels of size 4, prompts and first tokens
        _case(name="kernel4_96", do="prefill", mixer="kernel", k=4, batch=96, prompt=120, steps=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "small", "rollout", "prefill", "prefill", "ragged", "replicated", "mixers"))
    cache = rng.choice(("fp32", "fp32", "fp16"))
    if kind in ("decode", "small"):
        b = _log(rng, 1, 8192 if kind == "decode" else 2048)
        c = _case(model="mid" if kind == "decode" else "small", batch=b, cache=cache, prompt=rng.randint(8, 450))
        if rng.random() < 0.4:
            c.update(do="decode", logits=rng.random() < 0.5)
        else:
            c["steps"] = min(rng.randint(2, 24), max(2, 16384 // b))
        return c
    if kind == "rollout":
        if rng.random() < 0.6:
            return _case(do="decode", model="rl", batch=_log(rng, 512, 16384), prompt=rng.randint(8, 900), cache=cache,
                         select="topk", top_k=rng.randint(20, 100), temperature=round(rng.uniform(0.6, 1.0), 2))
        return _case(do="decode", model="rl", batch=_log(rng, 512, 6000), prompt=rng.randint(8, 900), cache=cache,
                     select="topp", top_p=round(rng.uniform(0.8, 0.95), 3), temperature=round(rng.uniform(0.6, 0.9), 2))
    if kind == "prefill":
        model = rng.choice(("mid", "mid", "small"))
        n = _log(rng, 8, 480 if model == "small" else 900)
        return _case(do="prefill", model=model, batch=_log(rng, 1, min(4096, 400000 // n)), prompt=n, cache=cache)
    if kind == "ragged":
        return _case(do="ragged", model=rng.choice(("mid", "small")), batch=_log(rng, 2, 256), prompt=rng.randint(16, 480),
                     steps=rng.randint(0, 8), cache=cache, logits=rng.random() < 0.5)
    if kind == "replicated":
        p = _log(rng, 1, 32)
        return _case(do="replicated", model="rl", prompts=p, batch=p * _log(rng, max(16, 512 // p + 1), 16384 // p),
                     prompt=rng.randint(16, 400), select="topk", temperature=0.8, cache=cache)
    mixer = rng.choice(("combined", "kernel", "head_proj"))
    return _case(do="prefill", mixer=mixer, k=rng.choice((2, 4, 8)) if mixer == "kernel" else 1, batch=_log(rng, 8, 700),
                 prompt=rng.randint(8, 160), steps=rng.randint(1, 6), cache=cache)


@functools.lru_cache(maxsize=2)
def _model(name, mixer, k, cache, flags=0):
    """The weights and the handle that a program keeps for as long as it runs."""
    s = MODELS[name]
    L, d, V, n, h, F = s["n_layers"], s["d_model"], s["vocab"], s["n_ctx"], s["n_heads"], s["ffn_mult"] * s["d_model"]
    g = torch.Generator(device="cuda").manual_seed(20 + L)

    def normal(*size, std=0.02, mean=0.0):
        return torch.randn(*size, generator=g, device="cuda").mul_(std).add_(mean)

    def decays(m, one):
        lam = 0.9 + 0.1 * torch.rand(m, generator=g, device="cuda")
        lam[one] = 1.0
        return lam

    def host(t):
        return t.cpu().numpy()

    E = normal(V, d, std=EMBED_STD)
    head = normal(V, d)
    for j, logit in enumerate(SUCCESSORS[name]):
        head += logit / (d * EMBED_STD * KEPT[name]) * torch.roll(E, j + 1, 0)
    w = {"E": host(E), "W_lm": host(head), "lnf_g": host(normal(d, mean=1.0)), "lnf_b": host(normal(d)), "layers": []}
    for _ in range(L):
        filters = k if mixer == "kernel" else h
        lw = dict(ln1_g=normal(d, mean=1.0), ln1_b=normal(d), alpha=normal(filters, n), beta=normal(n, d), lam=decays(filters, 0),
                  ln2_g=normal(d, mean=1.0), ln2_b=normal(d), W1=normal(F, d), b1=normal(F), W2=normal(d, F), b2=normal(d))
        if mixer == "combined":
            lw.update(alpha_col=normal(h, n), lam_col=decays(h, -1), w_comb=0.5 + 0.5 * torch.rand(h, 2, generator=g, device="cuda"))
        if mixer == "head_proj":
            lw.update(W_in=normal(d, d), W_out=normal(d, d))
        w["layers"].append({key: host(t) for key, t in lw.items()})
    shape = dict(s, mixer=mixer if mixer in ("combined", "kernel") else "mixed", kernel_size=k, head_proj=mixer == "head_proj")
    return srm.SRM(shape, w, device="cuda:0", state_dtype=cache, flags=flags)


def prepare(case, seed, flags=0):
    m = _model(case["model"], case["mixer"], case["k"], case["cache"], flags)
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, n, V = case["batch"], case["prompt"], m.cfg.vocab
    s = {"case": case, "model": m, "state": m.new_state(B),
         "sampling": srm.Sampling(case["select"], top_k=case["top_k"], temperature=case["temperature"], seed=seed, top_p=case["top_p"])}

    def tokens(*size):       # ids as in text: rank r about as often as 1 / r
        return torch.exp(torch.rand(*size, generator=g, device="cuda") * math.log(V)).to(torch.int32).sub_(1).clamp_(0, V - 1)

    st = s["state"]
    if case["do"] in ("decode", "generate"):
        s["workspace"] = m.new_workspace(min(B, 12288))
        s["tokens"] = tokens(B)
        st.last_token().copy_(s["tokens"])
        # the cache as a prompt leaves it: sums of alpha-weighted inputs (row-repeat) or of whole ones (column-repeat)
        for layer in range(m.cfg.n_layers):
            S = st.layer(layer)
            S.normal_(generator=g)
            if case["mixer"] == "combined":
                S[0] *= 0.1
                S[1] *= 3.0
            elif case["mixer"] == "kernel":
                S *= 3.0
            else:
                S[:, : m.cfg.d_model // 2] *= 0.1
                S[:, m.cfg.d_model // 2:] *= 3.0
        st.pos = n
        if case["select"] == "topk":       # every sample has been through a selection before
            m.decode_step(st, s["tokens"], s["sampling"], 0, s["workspace"])
    else:
        P = case["prompts"] or B
        need = max(m.workspace_bytes(min(B, 12288)), m.new_workspace(1, n, P).numel() + 256 * P + (
            m.cfg.n_layers * m.planes * m.cfg.d_model * 4 * P if case["do"] == "replicated" else 0))
        s["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
        s["tokens"] = tokens(P, n)
        if case["do"] == "ragged":
            s["lengths"] = torch.randint(max(1, n // 20), n + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
    if case["steps"]:
        s["out"] = torch.zeros(B, case["steps"], dtype=torch.int32, device="cuda")
    return s


def run(s):
    case, m, st, ws, samp = s["case"], s["model"], s["state"], s["workspace"], s["sampling"]
    out = {}
    if case["do"] == "decode":
        st.pos = case["prompt"]
        r = m.decode_step(st, s["tokens"], samp, 1, ws, want_logits=case["logits"])
    elif case["do"] == "generate":
        st.pos = case["prompt"]
        r = None
    else:
        st.reset()
        if case["do"] == "prefill":
            r = m.prefill(st, s["tokens"], samp, ws, want_logits=case["logits"])
        elif case["do"] == "ragged":
            r = m.prefill_ragged(st, s["tokens"], s["lengths"], samp, ws, want_logits=case["logits"])
        else:
            r = m.prefill_replicated(st, s["tokens"], st.B // case["prompts"], samp, ws, want_logits=case["logits"])
    if r is not None:
        out["token"], out["logits"] = r if case["logits"] else (r, None)
    if case["steps"]:
        out["generated"] = m.generate(st, case["steps"], 1, samp, ws, out=s["out"])
    out["cache"] = [st.layer(layer) for layer in range(m.cfg.n_layers)]
    return out


def work(case):
    s = MODELS[case["model"]]
    L, d, V, B, n = s["n_layers"], s["d_model"], s["vocab"], case["batch"], case["prompt"]
    per_row = L * (2 * s["ffn_mult"] * d * d + (2 * d * d if case["mixer"] == "head_proj" else 0))     # multiply-adds of the layers
    weights = 2 * (per_row + d * V)
    planes = {"combined": 2, "kernel": case["k"]}.get(case["mixer"], 1)
    cache = B * L * d * planes * (4 if case["cache"] == "fp32" else 2)
    logits = 4 * B * V if case["logits"] else 0
    steps = case["steps"] if case["do"] != "decode" else 1
    flops = steps * B * 2 * (per_row + d * V)
    passes, nbytes = steps, 2 * cache * steps + 4 * B * steps + logits
    if case["do"] not in ("decode", "generate"):
        P = case["prompts"] or B
        rows = P * n if case["do"] != "ragged" else P * (n + max(1, n // 20)) // 2
        flops += 2 * (rows * per_row + P * d * V)
        nbytes += cache + 4 * rows + 2 * d * min(rows, V)
        passes += 1
    nbytes += weights * (passes if weights > L2_BYTES else 1)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Measured between paths of the library that add in another order at the same precision (single-kernel step and
    # one kernel per operation, ranges of K and whole tiles, the two prefill mixers; all three models): at most 2.8e-3
    # on logits, 1.1e-3 on the cache, 0.0155 on a single value, and 1 sampled token of 700.
    return {"rel": 1e-2, "max": 0.06, "differ": 5e-3}
