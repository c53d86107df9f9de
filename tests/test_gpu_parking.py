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


@pytest.mark.parametrize("d,ff,nq,nkv,hd,vocab,n_prompt,n", SHAPES)
def test_parked_stages_leave_the_bits(d, ff, nq, nkv, hd, vocab, n_prompt, n):
    """Stages are parked, and a call without parking gives the same logits, bit for bit: one column and up to six."""
    cfg = config(d, ff, nq, nkv, hd, vocab)
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda"))
    for l in cfg.exit_layers:
        gm.set_exit_head(l, None, cfg.logit_scale)
    prompt = synth.make_prompt(cfg, n=n_prompt).numpy()
    for early in (0, 5):
        got = []
        for most in (2, 1, 0):
            S = binding.Session(gm, 1, n_prompt + n + 8, 64, 5)
            S.set_parking(most)
            S.capture_logits(n + 8)
            S.prefill(prompt)
            out = S.adaptive_decode(n, 0.0, cfg.exit_layers, early) if early else S.plain_decode(n)
            got.append((out[0], S.captured_logits()[:n].clone()))
            assert (S.parked() > 0) == (most > 0), (early, most)
        for out, logits in got[1:]:
            assert np.array_equal(out, got[0][0]) and torch.equal(logits, got[0][1]), early


def parkable(N, K, mode, most):
    """(most stages that the warps of all CTAs can park, whether all of them are sure to land): host arithmetic from the plans."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nch, pair, total = (K + 511) // 512, 2 if mode else 1, 0
    sure = most >= pair   # (a second matrix' stage that is not parked keeps its place in the ring)
    for cta in range(sms):
        p = binding.debug_gemm_plan(N, K, mode, sms, cta)
        ng = p["n"] if p["split"] else min(p["t1"] - p["t0"], 8)
        ts = 1 << max(ng - 1, 0).bit_length()
        ks = 8 // ts
        for slot in range(ng):
            chunks = list(range(nch))
            if p["split"] and slot == 0:
                chunks = [k for k in chunks if k < p["s0_pub_k1"] or k >= p["s0_own_k0"]]
            elif p["split"] and slot == ng - 1:
                chunks = chunks[:p["sl_k1"]]
            sure = sure and len(chunks) == nch   # a slot with a gap may find the ring full of other warps' third stages
            published = p["s0_pub_k1"] if p["split"] and slot == 0 else 0
            parts = [chunks[:published], chunks[published:]]
            for k in range(ks):
                total += min(sum(len(c[k::ks]) for c in parts) * pair, most)
    return total, sure


# one stage for one warp of a CTA; one for each; more than two for each; a pair of matrices, one chunk and many; several slots, some of them
# idle; tiles cut between CTAs, their first parts published; two groups of tiles
@pytest.mark.parametrize("N,K,mode", [(148 * 16, 512, 0), (148 * 16, 4096, 0), (148 * 16, 14336, 0), (2 * 148 * 16, 512, 1), (2 * 148 * 16, 4096, 1),
                                      (148 * 16 * 5, 1216, 0), (6144, 4096, 0), (2 * 5504, 2048, 1), (24000, 576, 0), (1000, 192, 0)])
@pytest.mark.parametrize("cols", [1, 4, 5, 8])
def test_products_from_parked_stages(N, K, mode, cols):
    W = synth.normal_tensor(5, 11, (N, K), 0.05, torch.bfloat16, "cuda")
    X = synth.normal_tensor(5, 12, (cols, K), 1.0, torch.float32, "cuda")
    ref, none = binding.debug_gemm_parked(W, X, mode, most=0, hold_ns=200_000)
    assert none == 0
    for most in (1, 2):
        Y, parked = binding.debug_gemm_parked(W, X, mode, most=most, hold_ns=200_000)   # (a stage lands within 2 us)
        total, sure = parkable(N, K, mode, most)
        assert 0 < parked <= total and (parked == total or not sure), (most, parked, total)
        assert torch.equal(Y, ref), most
    assert torch.equal(binding.debug_gemm(W, X, mode)[0], ref)
    # the activations come after the consumers have given up: parked stages are multiplied with whatever is there, and the call says so
    with pytest.raises(binding.AdaError) as e:
        binding.debug_gemm_parked(W, X, mode, hold_ns=400_000, wait_ns=100_000)
    assert e.value.code == -5
    assert torch.equal(binding.debug_gemm_parked(W, X, mode)[0], ref)
