"""fp32 decoding in one launch (csrc/resident.cuh) against the per-operation kernels, which take the sessions that do not
qualify for it: here one with room for sixteen early tokens."""

import numpy as np
import pytest
import torch

from paper_2506_03700_b200 import binding, synth

pytestmark = pytest.mark.gpu


def decode(gm, cfg, prompts, n, early, max_early, mode):
    S = binding.Session(gm, len(prompts), max(len(p) for p in prompts) + n + 8, 16, max_early)
    S.capture_logits(n)
    for i, p in enumerate(prompts):
        S.prefill(p, seq=i)
    if mode == "plain":
        out = S.plain_decode(n)
    else:
        if mode == "tape":   # exits against the heads' own decisions, so that tokens are rejected and the cache rolled back
            S.set_exit_tape([1, 1, 0, 1, 2, 1, 1, 1, 0, 0, 1] * 6)
        out = S.adaptive_decode(n, 0.3, cfg.exit_layers, early)
    return out, S.captured_logits().cpu().numpy().astype(np.float64)


# (q heads, kv heads, head_dim, width, d_ff, vocabulary): one and several 16-byte pieces per lane, ragged ones, rows of 768
# elements and more (the weights of a row in several pieces; prompt passes of fewer rows), an odd vocabulary; narrower than the
# GPU has SMs
SHAPES = [(4, 4, 64, 256, 688, 2048), (6, 2, 32, 192, 328, 1001), (2, 1, 128, 256, 800, 515), (4, 1, 32, 1032, 136, 300),
          (4, 2, 32, 128, 344, 1024), (2, 2, 32, 64, 128, 600), (1, 1, 32, 24, 40, 256)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("lens,early,mode", [((1,), 5, "plain"), ((31,), 5, "adaptive"), ((33,), 1, "tape"), ((127,), 5, "tape"),
                                              ((130, 5, 64), 3, "adaptive"), ((40, 9, 17, 32, 1, 3, 8, 2), 5, "tape")])
def test_one_launch_equals_the_per_operation_path(shape, lens, early, mode):
    nq, nkv, hd, d, dff, vocab = shape
    cfg = synth.small_config(n_layers=4, d_model=d, n_q_heads=nq, n_kv_heads=nkv, head_dim=hd, d_ff=dff, vocab=vocab, sigma=0.08,
                             resid_scale=0.5, exit_layers=(1, 3))
    w = synth.make_weights(cfg, device="cuda", norm_gain_jitter=0.2)
    gm = binding.Model(cfg, w)
    gm.set_exit_head(1, synth.make_head_transform(cfg, 1, device="cuda", noise=0.1), 4.0)
    gm.set_exit_head(3, None, 4.0)
    prompts = [synth.make_prompt(cfg, n=k, seq=i).numpy() for i, k in enumerate(lens)]
    n = 20
    out, lg = decode(gm, cfg, prompts, n, early, 5, mode)
    ref, lr = decode(gm, cfg, prompts, n, early, 15 if len(lens) == 8 else 16, mode)
    assert lg.shape == lr.shape
    # The same fp32 products summed in another order.  Rounding of a sum of up to 1032 products: 6e-8 x sqrt(1032) = 2e-6 of its
    # size; some 28 products one after the other: 1e-5; both sides and the largest of 6000 logits (four standard deviations):
    # 6e-5 of the logits' spread.  Asserted: the bound that fp32 logits are held to against the oracle.
    tol = 1e-4 * lr.std()
    top = np.sort(lr, axis=-1)
    clear = (top[:, -1] - top[:, -2]) > 2 * tol
    stop = int(np.argmin(clear)) if not clear.all() else n
    assert stop > 3, "the synthetic logits leave nothing to compare"
    assert np.abs(lg[:stop] - lr[:stop]).max() <= tol
    assert np.array_equal(out[0][:stop], ref[0][:stop])
    for s in range(1, len(lens)):   # the other sequences' logits are not kept: their tokens
        assert np.array_equal(out[s], ref[s])


# fp32 in one launch; fp32 and bf16 in one launch per operation (room for sixteen early tokens; 96 features a head); the bf16 kernel
@pytest.mark.parametrize("dtype,hd,max_early", [("fp32", 64, 5), ("fp32", 64, 16), ("bf16", 96, 5), ("bf16", 64, 5)])
def test_tokens_stay_in_the_vocabulary_where_no_logit_is_a_number(dtype, hd, max_early):
    """The argmax of logits that are all NaN is none; what is emitted, and read back as an embedding row, is a token all the same,
    the one after the prompt included."""
    cfg = synth.small_config(dtype=dtype, n_layers=3, d_model=256, n_q_heads=2, n_kv_heads=1, head_dim=hd, d_ff=320, vocab=500,
                             exit_layers=(1, 2))
    w = synth.make_weights(cfg, device="cuda", tied=False)
    w["lm_head"].fill_(float("nan"))
    gm = binding.Model(cfg, w)
    for l in cfg.exit_layers:
        gm.set_exit_head(l, None, 4.0)
    S = binding.Session(gm, 2, 64, 64, max_early)
    for mode in ("plain", "adaptive"):
        for i, n in enumerate((5, 12)):
            S.prefill(synth.make_prompt(cfg, n=n, seq=i).numpy(), seq=i)
        out = S.plain_decode(6) if mode == "plain" else S.adaptive_decode(6, 0.1, cfg.exit_layers, 5)
        assert out.min() >= 0 and out.max() < cfg.vocab


@pytest.mark.parametrize("batch,max_early", [(16, 2), (9, 4)])
def test_heads_over_more_than_eight_rows_give_each_sequence_its_own_bits(batch, max_early):
    """More than eight newest tokens at an intermediate head: a row's probability does not depend on its company.  (Without early
    exits every step evaluates every sequence at every exit layer; the log holds them in that order.)"""
    cfg = synth.small_config(n_layers=4, d_model=256, n_q_heads=4, n_kv_heads=4, head_dim=64, d_ff=688, vocab=2048, sigma=0.08,
                             resid_scale=0.5, exit_layers=(1, 3))
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda", norm_gain_jitter=0.2))
    for l in cfg.exit_layers:
        gm.set_exit_head(l, None, 4.0)
    prompts = [synth.make_prompt(cfg, n=5 + i, seq=i).numpy() for i in range(batch)]

    def run(ps):
        S = binding.Session(gm, len(ps), 64, 16, max_early)
        S.capture_heads()
        for i, p in enumerate(ps):
            S.prefill(p, seq=i)
        out = S.adaptive_decode(20, 2.0, cfg.exit_layers, max_early)
        return out, S.captured_heads()[:, 2:].reshape(-1, len(ps), 2).copy()   # (token, p) by step and layer, sequence

    out, log = run(prompts)
    assert len(log) >= 30
    for i, p in enumerate(prompts):
        o, l = run([p])
        assert np.array_equal(o[0], out[i])
        assert np.array_equal(l[:, 0], log[:, i]), i


@pytest.mark.parametrize("during", ["prompt", "decode"])
def test_a_wait_that_runs_out_ends_the_call_with_a_timeout_and_the_session_recovers(during):
    """Values pass between the CTAs as words that the readers wait for, with a limit.  Set far below the time that a word takes, the
    first wait that is not satisfied at once gives up, the others follow, and the call returns ADA_ETIMEOUT.  After a reset and
    a prompt the session gives what a fresh one gives."""
    cfg = synth.small_config(n_layers=4, d_model=256, n_q_heads=4, n_kv_heads=4, head_dim=64, d_ff=688, vocab=2048, sigma=0.08,
                             resid_scale=0.5, exit_layers=(1, 3))
    plan = binding.debug_resident_plan(cfg, 2, 5)
    assert plan["rows"] > 0 and plan["prompts"]
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda", norm_gain_jitter=0.2))
    gm.set_exit_head(1, synth.make_head_transform(cfg, 1, device="cuda", noise=0.1), 4.0)
    gm.set_exit_head(3, None, 4.0)
    prompts = [synth.make_prompt(cfg, n=k, seq=i).numpy() for i, k in enumerate((40, 12))]
    n = 16

    def whole(S):
        for i, p in enumerate(prompts):
            S.prefill(p, seq=i)
        return S.adaptive_decode(n, 0.3, cfg.exit_layers, 5), S.captured_logits().cpu().numpy().copy()

    def session():
        S = binding.Session(gm, 2, 96, 16, 5)
        S.capture_logits(n)
        return S

    ref, lr = whole(session())
    S = session()
    if during == "decode":
        for i, p in enumerate(prompts):
            S.prefill(p, seq=i)
    S.set_wait_limit(20)                  # nanoseconds
    with pytest.raises(binding.AdaError) as e:
        S.prefill(prompts[0], seq=0) if during == "prompt" else S.adaptive_decode(n, 0.3, cfg.exit_layers, 5)
    assert e.value.code == -5
    torch.cuda.synchronize()              # the context is intact
    S.set_wait_limit(2_000_000_000)
    S.reset()
    out, lg = whole(S)
    assert np.array_equal(out, ref) and np.array_equal(lg, lr)
