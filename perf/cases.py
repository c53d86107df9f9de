"""What the decode library is measured on: whole requests through its public calls.

A pass takes one request (or a batch of them) from its prompt to its generated tokens: `ada_prefill` for every
sequence, then one decode call, through the binding's `Session`.  It returns the tokens and the final logits of
every generated token of the first sequence.  The shapes are the configurations in `synth.CONFIGS` (the fp32 tiny
decoder and the 1B, 8B and 13B shaped bf16 decoders), at full depth and width; prompts run from a few tokens to
8192, generations from one token to a few hundred, sessions hold one to eight sequences and up to five early
predictions in flight (the paper's cap).

Weights.  Layer matrices are N(0, 0.02^2) with the output projections scaled as each configuration says.  A trained
model is confident about most next tokens and its heads at intermediate layers mostly agree with its last layer;
plain random heads are neither.  So for the bf16 shapes the embedding carries a signal that outlives the layers
and the LM head maps every token to one successor: the decoder runs through a fixed random cycle of tokens with a
clear margin, while every other logit is made of what the layers computed.  An intermediate head's dense
transformation T sees half of the features only, and for one token in ten a decoy wins on that half: a confident
early prediction that the verification has to reject (the paper reports about one in twenty).
"""

import numpy as np
import torch

from paper_2506_03700_b200 import binding, synth

DECOYS = 0.1          # share of the tokens whose early prediction through T is wrong
# Embedding scale of each shape: the residual noise that its layers add has 4/3 of this size at the last layer.
EMBED_SCALE = {"1b": 0.5, "8b": 1.5, "13b": 2.6}


def listed():
    return [
        # The tiny fp32 decoder as configured (16 + 128 tokens, heads after layers 2 and 3): a small model where latency counts.
        dict(name="tiny-fp32-adaptive", model="tiny", mode="adaptive", batch=1, max_early=5, prompt_lo=16, prompt_hi=16, tokens=128, T=False),
        # A short exchange with the 1B shape, plain greedy decoding.
        dict(name="1b-chat-plain", model="1b", mode="plain", batch=1, max_early=5, prompt_lo=45, prompt_hi=45, tokens=48, T=False),
        # The configured 512-token prompt of the 1B shape, adaptive with trained-like dense heads.
        dict(name="1b-adaptive", model="1b", mode="adaptive", batch=1, max_early=5, prompt_lo=512, prompt_hi=512, tokens=128, T=True),
        # Sampled decoding with stochastic verification.
        dict(name="1b-sampled", model="1b", mode="sampled", batch=1, max_early=4, prompt_lo=203, prompt_hi=203, tokens=64, T=True),
        # Eight users of one session, prompts of different lengths, plain decoding over one weight stream.
        dict(name="1b-batch8-plain", model="1b", mode="plain", batch=8, max_early=0, prompt_lo=64, prompt_hi=300, tokens=48, T=False),
        # A question of one line: too short for the block-wise prompt pass.
        dict(name="8b-question", model="8b", mode="adaptive", batch=1, max_early=5, prompt_lo=21, prompt_hi=21, tokens=32, T=True),
        # The main configuration: 1024-token prompt, a long answer with up to five early tokens in flight.
        dict(name="8b-adaptive", model="8b", mode="adaptive", batch=1, max_early=5, prompt_lo=1024, prompt_hi=1024, tokens=128, T=True),
        # Classification or a tool call: a prompt of odd length and two tokens of answer.
        dict(name="8b-classify", model="8b", mode="plain", batch=1, max_early=5, prompt_lo=777, prompt_hi=777, tokens=2, T=False),
        # The long-context configuration's prompt: summarising a document of 8000 tokens.
        dict(name="8b-document", model="8b", mode="plain", batch=1, max_early=5, prompt_lo=8000, prompt_hi=8000, tokens=12, T=False),
        # Generation over a context of some thousand tokens, untransformed heads (T = I).
        dict(name="8b-long-adaptive", model="8b", mode="adaptive", batch=1, max_early=5, prompt_lo=3000, prompt_hi=3000, tokens=96, T=False),
        # Four independent sequences on the 13B shape with ragged prompts, one early token each.
        dict(name="13b-batch4-early1", model="13b", mode="adaptive", batch=4, max_early=1, prompt_lo=256, prompt_hi=500, tokens=32, T=True),
        # The same with the paper's five early tokens in flight per sequence.
        dict(name="13b-batch4-early5", model="13b", mode="adaptive", batch=4, max_early=5, prompt_lo=256, prompt_hi=500, tokens=16, T=True),
    ]


# Most prompt tokens and most generated tokens of a drawn case, over all its sequences.
_MOST = {"tiny": (512, 256), "1b": (8192, 384), "8b": (8192, 160), "13b": (2000, 72)}


def draw(rng):
    model = rng.choice(["tiny", "1b", "1b", "8b", "8b", "13b"])
    mode = rng.choice(["plain", "adaptive"] if model == "tiny" else ["plain", "adaptive", "adaptive", "sampled"])
    batch = 1 if rng.random() < 0.6 else rng.randint(2, 4 if model == "13b" else 8)
    most_p, most_t = _MOST[model]
    hi = int(round(9 * (most_p / batch / 9) ** rng.random()))
    lo = max(1, int(hi * rng.uniform(0.4, 1.0))) if batch > 1 else hi
    # what the prompts leave of the cost of the largest listed case goes to generation
    left = max(2.0, most_t / batch * (1.0 - hi * batch / (1.15 * most_p)))
    tokens = max(1, int(round(left ** rng.random())))
    early = rng.randint(0 if mode == "plain" else 1, 5)
    return dict(model=model, mode=mode, batch=batch, max_early=early, prompt_lo=lo, prompt_hi=hi, tokens=tokens,
                T=bool(mode != "plain" and model != "tiny" and rng.random() < 0.7))


def _prompt_lengths(case):
    """Lengths of the sequences' prompts, spread over [prompt_lo, prompt_hi]."""
    lo, hi = case["prompt_lo"], case["prompt_hi"]
    return [lo + int((hi - lo) * ((0.618034 * (k + 1)) % 1.0) + 0.5) for k in range(case["batch"])]


def _peaked_weights(cfg, embed_scale, gen):
    """Weights of a decoder that walks a cycle of tokens with confidence; (weights, tokens of the cycle)."""
    dt, d, v = cfg.torch_dtype, cfg.d_model, cfg.vocab

    def normal(rows, cols, sigma):
        return torch.empty(rows, cols, dtype=dt, device="cuda").normal_(0.0, sigma, generator=gen)

    w = {}
    unit = normal(v, d, 1.0)
    ids = torch.randperm(v, device="cuda", generator=gen)
    n_decoy = int(v * DECOYS)
    decoy, cycle = ids[:n_decoy], ids[n_decoy:]
    fooled = cycle[torch.randperm(len(cycle), device="cuda", generator=gen)[:n_decoy]]
    head = torch.empty_like(unit)
    head[torch.roll(cycle, -1)] = unit[cycle] * cfg.sigma          # the successor of cycle[i] is cycle[i + 1]
    head[decoy, :d // 2] = unit[fooled, :d // 2] * (1.5 * cfg.sigma)   # wins on the half that T keeps, loses on both
    head[decoy, d // 2:] = unit[fooled, d // 2:] * -cfg.sigma
    unit[decoy] = unit[cycle[:n_decoy]]                            # a decoy that was emitted early goes on like a token of the cycle
    w["tok_embed"], w["lm_head"] = unit.mul_(embed_scale), head
    w["final_norm"] = torch.ones(d, dtype=dt, device="cuda")
    for l in range(cfg.n_layers):
        p = "layers.%d." % l
        w[p + "attn_norm"] = torch.ones(d, dtype=dt, device="cuda")
        w[p + "ffn_norm"] = torch.ones(d, dtype=dt, device="cuda")
        w[p + "wqkv"] = normal(cfg.qkv_rows, d, cfg.sigma)
        w[p + "wo"] = normal(d, cfg.n_q_heads * cfg.head_dim, cfg.sigma * cfg.resid_scale)
        w[p + "w_gate_up"] = normal(2 * cfg.d_ff, d, cfg.sigma)
        w[p + "w_down"] = normal(d, cfg.d_ff, cfg.sigma * cfg.resid_scale)
    return w, cycle


def prepare(case, seed):
    cfg = synth.CONFIGS[case["model"]]
    lens = _prompt_lengths(case)
    rng = np.random.default_rng(seed)
    if case["model"] == "tiny":
        weights = synth.make_weights(cfg, seed=seed, device="cuda")
        prompts = [rng.integers(0, cfg.vocab, n).astype(np.int32) for n in lens]
    else:
        gen = torch.Generator(device="cuda").manual_seed(seed)
        weights, cycle = _peaked_weights(cfg, EMBED_SCALE[case["model"]], gen)
        cycle = cycle.cpu().numpy()
        prompts = [cycle[rng.integers(0, len(cycle), n)].astype(np.int32) for n in lens]
    model = binding.Model(cfg, weights)
    if case["mode"] != "plain":
        T = None
        if case["T"]:
            keep = torch.zeros(cfg.d_model, device="cuda")
            keep[:cfg.d_model // 2] = 1.0
            T = torch.diag(keep).to(cfg.torch_dtype)
        for layer in cfg.exit_layers:
            model.set_exit_head(layer, T, cfg.logit_scale)
    n = case["tokens"]
    max_seq = max(lens) + n + 8
    session = binding.Session(model, case["batch"], max_seq, 64, case["max_early"])
    session.capture_logits(n)
    state = dict(case=case, cfg=cfg, session=session, prompts=prompts)
    if case["mode"] == "sampled":
        state["uniforms"] = rng.random((case["batch"], max_seq, binding.SAMPLE_NU), dtype=np.float32)
    return state


def run(state):
    case, cfg, s = state["case"], state["cfg"], state["session"]
    for i, p in enumerate(state["prompts"]):
        s.prefill(p, seq=i)
    n, early = case["tokens"], case["max_early"]
    if case["mode"] == "plain":
        tokens = s.plain_decode(n)
    elif case["mode"] == "adaptive":
        tokens = s.adaptive_decode(n, cfg.threshold, cfg.exit_layers, early)
    else:
        tokens = s.sampling_decode(n, 0.7, cfg.threshold, cfg.exit_layers, early, state["uniforms"])
    return {"tokens": tokens, "logits": s.captured_logits()}


def work(case):
    """Weights and cache rows that the prompts and every step have to read, multiply-adds of one bf16 (fp32) product."""
    cfg = synth.CONFIGS[case["model"]]
    size = 4 if cfg.dtype == "fp32" else 2
    lens, n, batch, L = _prompt_lengths(case), case["tokens"], case["batch"], cfg.n_layers
    d, qd, kvd = cfg.d_model, cfg.n_q_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim
    layer = (qd + 2 * kvd) * d + qd * d + 3 * cfg.d_ff * d
    head, t_mat = cfg.vocab * d, d * d if case["T"] else 0
    flops = sum(2.0 * L * layer * p + 2.0 * L * qd * p * p + 2.0 * head for p in lens)
    cache = sum(2.0 * L * kvd * p for p in lens)      # elements of K and V of all sequences
    weights, steps = 0.0, 0.0                         # elements streamed by the decode steps; steps that read the whole cache
    if case["mode"] == "plain":
        weights, steps = (n - 1.0) * (L * layer + head), n - 1.0
        flops += 2.0 * (n - 1) * batch * (L * layer + head)
    else:   # every early token accepted: max_early exits at the first exit layer, then one step to the last
        first = cfg.exit_layers[0]
        cycles, k = (n - 1.0) / (case["max_early"] + 1), case["max_early"]
        weights = cycles * (k * (first * layer + t_mat + head) + L * layer + head)
        steps = cycles * (k * first / L + 1.0)
        flops += 2.0 * batch * ((n - 1) * L * layer + (n - 1) * head + cycles * k * (t_mat + head))
    if (L * layer + head) * size < 64e6:
        weights = 0.0                                 # such a model stays in the L2 cache: each weight is read once
    nbytes = size * (L * layer + head + 2.0 * cache + weights + steps * cache) + 4.0 * n * cfg.vocab
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Relative error of the logits.  fp32: 1.7e-7 against the double-precision oracle; another order of the sums moves
    # them as much.  bf16: the prompt through the decode kernel (eight positions a pass) instead of the block-wise pass,
    # i.e. other summation orders in front of the cache's bf16 rounding, moves them by 0.4e-4 to 1.8e-4 (1B, 8B) and
    # 3.8e-4 (13B).  The tokens do not depend on either: the smallest gap between the two highest logits is 7 (tiny) and
    # 14 (others) standard deviations.
    return {"rel": 2e-6} if case["model"] == "tiny" else {"rel": 2e-3}
