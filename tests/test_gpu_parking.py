"""Decode products whose weight stages are parked in tensor memory, and rows with one or several attention chunks, at the edges:
depths of one ragged chunk, exactly one, one more than a CTA's warps, heads of one and of many tile groups; contexts that end below,
at and above a chunk.  Tolerances as in test_gpu_persistent (logits within 2e-2 x their std of the double-precision oracle;
adaptive decoding, which puts one to six columns through the same products, bit-exact with plain)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2506_03700_b200 import binding, synth
from test_gpu_parity import Pair, check_against_oracle

# d_model, d_ff, q heads, kv heads, head_dim, vocab, prompt, tokens
SHAPES = [(64, 64, 1, 1, 64, 130, 3, 12),           # products of one ragged chunk and four tiles: most CTAs and warps own nothing
          (512, 512, 4, 1, 128, 1000, 126, 6),      # exactly one chunk; the context passes 128 positions while decoding
          (576, 4224, 8, 2, 64, 2400, 20, 10),      # two chunks, the second ragged; nine chunks: one warp owns two stages
          (1024, 2752, 8, 8, 128, 24000, 255, 5)]   # eleven tiles of the head a CTA: two groups; the third attention chunk begins


def config(d, ff, nq, nkv, hd, vocab):
    return synth.small_config(name="park", dtype="bf16", n_layers=3, d_model=d, n_q_heads=nq, n_kv_heads=nkv, head_dim=hd, d_ff=ff, vocab=vocab,
                              sigma=0.05, resid_scale=0.6, exit_layers=(1, 2), rope_base=10000.0)


@pytest.mark.parametrize("d,ff,nq,nkv,hd,vocab,n_prompt,n", SHAPES)
def test_edges_of_products_and_chunks(d, ff, nq, nkv, hd, vocab, n_prompt, n):
    cfg = config(d, ff, nq, nkv, hd, vocab)
    pair = Pair(cfg)
    prompt = synth.make_prompt(cfg, n=n_prompt).numpy()

    def decode(run):
        S = binding.Session(pair.gm, 1, n_prompt + n + 8, 64, 5)
        assert S.get_path() == 1
        S.capture_logits(n + 8)
        S.prefill(prompt)
        return run(S)[0], S.captured_logits()[:n].clone()

    tokens, logits = decode(lambda S: S.plain_decode(n))
    check_against_oracle(pair, prompt, tokens, logits.cpu().numpy())
    for gamma in (0.0, 0.3):
        out, lg = decode(lambda S: S.adaptive_decode(n, gamma, cfg.exit_layers, 5))
        assert np.array_equal(out, tokens) and torch.equal(lg, logits), gamma


@pytest.mark.parametrize("batch,early", [(3, 1), (8, 0), (2, 5)])   # six and eight columns of one tile; 24 columns
def test_columns_of_several_sequences(batch, early):
    cfg = config(576, 4224, 8, 2, 64, 2400)
    pair = Pair(cfg)
    n = 9
    prompts = [synth.make_prompt(cfg, n=118 + 5 * s, seq=s).numpy() for s in range(batch)]   # some below one chunk, some above

    def decode(ps):
        S = binding.Session(pair.gm, len(ps), 256, 64, early)
        for s, p in enumerate(ps):
            S.prefill(p, seq=s)
        return S.adaptive_decode(n, 0.2, cfg.exit_layers, early) if early else S.plain_decode(n)

    together = decode(prompts)
    for s, p in enumerate(prompts):
        assert np.array_equal(together[s], decode([p])[0]), s


@pytest.mark.parametrize("batch,early", [(1, 5), (3, 1), (2, 5)])   # one sequence; six columns of one tile; 24 columns
def test_waits_that_run_out_anywhere(batch, early):
    """Limits from far below what a wait lasts to about as long as a phase: which wait gives up first, in which lane, with stages
    parked or not and at a control point or not, differs from run to run.  Every call ends with a time-out or with the right tokens,
    and the session decodes correctly afterwards."""
    cfg = config(576, 4224, 8, 2, 64, 2400)
    pair = Pair(cfg)
    n = 9
    prompts = [synth.make_prompt(cfg, n=118 + 5 * s, seq=s).numpy() for s in range(batch)]
    S = binding.Session(pair.gm, batch, 256, 64, early)

    def decode(limit):
        S.set_wait_limit(2_000_000_000)
        S.reset()
        for s, p in enumerate(prompts):
            S.prefill(p, seq=s)
        S.set_wait_limit(limit)
        return S.adaptive_decode(n, 0.2, cfg.exit_layers, early)

    ref = decode(2_000_000_000)
    ran_out = 0
    for limit in (50, 400, 1500, 3000, 6000, 12000, 40000):
        try:
            assert np.array_equal(decode(limit), ref), limit
        except binding.AdaError as e:
            assert e.code == -5, limit
            ran_out += 1
            torch.cuda.synchronize()      # the context is intact
        assert np.array_equal(decode(2_000_000_000), ref), limit
    assert ran_out > 0
