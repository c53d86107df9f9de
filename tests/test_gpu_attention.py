"""Decode attention at the edges of its 64-position sub-blocks and 128-position chunks, with one and with two query tiles in
use, against the per-operation kernels; and the same bits whichever of the two it is."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2506_03700_b200 import binding, synth


@pytest.mark.parametrize("head_dim,nq,nkv", [(64, 8, 2), (128, 4, 1), (64, 6, 2), (128, 4, 2), (64, 3, 3)])
def test_chunk_edges(head_dim, nq, nkv):
    cfg = synth.small_config(dtype="bf16", n_layers=3, d_model=256, n_q_heads=nq, n_kv_heads=nkv, head_dim=head_dim, d_ff=704,
                             vocab=1024, sigma=0.08, resid_scale=0.8, exit_layers=(1, 2))
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda"))
    for l in cfg.exit_layers:
        gm.set_exit_head(l, None, cfg.logit_scale)
    n = 6
    for n_prompt in (1, 59, 62, 64, 121, 126, 128, 250, 255, 700):
        prompt = synth.make_prompt(cfg, n=n_prompt).numpy()
        got = []
        for how in ("plain", "adaptive", "per-operation", "per-operation prompt"):
            S = binding.Session(gm, 1, 768, 64, 5)
            S.set_prefill(False)
            if how == "per-operation prompt":
                S.set_path(0)
            S.capture_logits(n + 4)
            S.prefill(prompt)
            if how == "per-operation":
                S.set_path(0)
            out = S.adaptive_decode(n, 0.0, cfg.exit_layers, 5) if how == "adaptive" else S.plain_decode(n)
            got.append((out[0], S.captured_logits()[:n].cpu().numpy()))
        (tp, lp), (ta, la), *others = got
        # every token leaves early (threshold 0), up to six columns in flight: the same bits as one column at a time
        assert np.array_equal(tp, ta) and np.array_equal(lp, la), n_prompt
        # Against the per-operation kernels, decoding on the same cache of the prompt and on their own: what differs are bf16
        # roundings of K and V (2^-9 of a value each).  Row i of the logits has seen tokens 0 .. i - 1 and was decoded for i > 0,
        # so the first row behind the last equal token still counts, and there always is one.
        for (to, lo), first in zip(others, (1, 0)):
            same = int(np.argmin(np.append(tp == to, False)))
            assert first == 0 or same >= 1, n_prompt   # (the first token comes out of the same prompt pass)
            for i in range(first, min(same + 1, n)):
                assert np.linalg.norm(lp[i] - lo[i]) <= 5e-3 * np.linalg.norm(lo[i]), (n_prompt, i)


@pytest.mark.parametrize("head_dim,nq,nkv", [(64, 8, 2), (128, 4, 1), (128, 4, 2), (64, 3, 3)])
def test_decode_attention_against_a_plain_softmax(head_dim, nq, nkv):
    """The logits of every decoded token against a float64 forward pass over the cache rows that the library holds: nothing that
    one- and two-tile attention share can hide."""
    cfg = synth.small_config(dtype="bf16", n_layers=2, d_model=256, n_q_heads=nq, n_kv_heads=nkv, head_dim=head_dim, d_ff=704,
                             vocab=1024, sigma=0.08, resid_scale=0.8, exit_layers=(1,))
    w = synth.make_weights(cfg, device="cuda")
    gm = binding.Model(cfg, w)
    W = {k: t.double().cpu().numpy() for k, t in w.items()}
    qd, kvd, half = nq * head_dim, nkv * head_dim, head_dim // 2
    rms = lambda x: x / np.sqrt((x * x).mean(-1, keepdims=True) + np.float32(cfg.rms_eps))
    n = 4
    for n_prompt in (1, 61, 127, 128, 253, 700):
        prompt = synth.make_prompt(cfg, n=n_prompt).numpy()
        S = binding.Session(gm, 1, 768, 64, 5)
        S.capture_logits(n + 4)
        S.prefill(prompt)
        tokens = np.concatenate([prompt, S.plain_decode(n)[0]])
        logits = S.captured_logits()[:n].cpu().numpy()
        kv = [[np.stack([S.read_kv(which, l, p) for p in range(n_prompt + n - 1)]).astype(np.float64) for which in (0, 1)] for l in range(cfg.n_layers)]
        for i in range(1, n):                       # row i: the pass of the token at position n_prompt + i - 1
            pos = n_prompt + i - 1
            x = W["tok_embed"][tokens[pos]]
            angle = pos * cfg.rope_base ** (-2.0 * np.arange(half) / head_dim)
            for l in range(cfg.n_layers):
                p = "layers.%d." % l
                q = (W[p + "wqkv"][:qd] @ (rms(x) * W[p + "attn_norm"])).reshape(nq, head_dim)
                z = (q[:, :half] + 1j * q[:, half:]) * np.exp(1j * angle)
                q = np.concatenate([z.real, z.imag], -1)
                k, v = (np.repeat(t[:pos + 1].reshape(pos + 1, nkv, head_dim), nq // nkv, 1) for t in kv[l])
                s = np.einsum("hd,thd->ht", q, k) / np.sqrt(head_dim)
                s = np.exp(s - s.max(-1, keepdims=True))
                x = x + W[p + "wo"] @ np.einsum("ht,thd->hd", s / s.sum(-1, keepdims=True), v).reshape(qd)
                gu = W[p + "w_gate_up"] @ (rms(x) * W[p + "ffn_norm"])
                g, u = gu[:cfg.d_ff], gu[cfg.d_ff:]
                x = x + W[p + "w_down"] @ (g / (1.0 + np.exp(-g)) * u)
            ref = W["tok_embed"] @ (rms(x) * W["final_norm"])
            # the cache is given, so only the splits into two bf16 parts (2^-17 of a value) and fp32 sums remain; six products deep
            assert np.linalg.norm(logits[i] - ref) <= 6e-5 * np.linalg.norm(ref), (n_prompt, i)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("batch,max_early", [(1, 5), (3, 5)])
def test_calls_pay_for_the_positions_they_reach_not_for_the_sessions_length(dtype, batch, max_early):
    """Short calls whose context grows over chunk boundaries (the layout of the chunk partials changes with it), in a session of
    512 positions and in one of 32768: the same bits, and the same bytes cleared."""
    cfg = synth.small_config(dtype=dtype, n_layers=3, d_model=256, n_q_heads=8, n_kv_heads=4, head_dim=64, d_ff=704, vocab=1024,
                             sigma=0.08, resid_scale=0.8, exit_layers=(1, 2))
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda"))
    for l in cfg.exit_layers:
        gm.set_exit_head(l, None, 4.0)
    got = []
    for max_seq in (512, 32768):
        S = binding.Session(gm, batch, max_seq, 64, max_early, kv_pages=8 * batch)
        S.capture_logits(64)
        seen, cleared = [], []
        for first in (5, 120):   # (a prompt of the decode kernel's passes, one of the dense pass where there is one)
            for i in range(batch):
                S.prefill(synth.make_prompt(cfg, n=first + 3 * i, seq=i).numpy(), seq=i)
                cleared.append(S.cleared_bytes())
            for n in (1, 7, 3, 20):
                seen.append(S.adaptive_decode(n, 0.2, cfg.exit_layers, max_early))
                cleared.append(S.cleared_bytes())
            seen.append(S.captured_logits().cpu().numpy().copy())
        got.append((seen, cleared))
    assert all(np.array_equal(a, b) for a, b in zip(got[0][0], got[1][0]))
    assert got[0][1] == got[1][1]
    assert got[0][1][-1] > got[0][1][batch + 1] > 0   # (the last call reaches a second chunk, the first of several tokens does not)


@pytest.mark.parametrize("head_dim,nq,nkv,batch", [(64, 8, 2, 1), (128, 4, 4, 1), (64, 8, 8, 3)])
def test_rows_written_in_a_launch_reach_the_chunks_of_its_later_steps(head_dim, nq, nkv, batch):
    """A chunk that the context has just left is read by bulk copies that wait for no barrier of their own step.  Its rows were written
    in earlier steps, by other CTAs: in the same launch here, in launches of their own (one step each) for what is compared, so that
    the end of a kernel orders them.  The same bits: prompts through the decode path, plain and adaptive decoding, across several chunks."""
    cfg = synth.small_config(dtype="bf16", n_layers=3, d_model=512, n_q_heads=nq, n_kv_heads=nkv, head_dim=head_dim, d_ff=704,
                             vocab=1024, sigma=0.08, resid_scale=0.8, exit_layers=(1, 2))
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda"))
    for l in cfg.exit_layers:
        gm.set_exit_head(l, None, cfg.logit_scale)
    n = 20
    for n_prompt in (120, 247, 377):
        prompts = [synth.make_prompt(cfg, n=n_prompt - 3 * s, seq=s).numpy() for s in range(batch)]
        for early in (0, 1):
            got = []
            for steps in (256, 1):
                S = binding.Session(gm, batch, 512, 64, early)
                S.set_prefill(False)
                S.set_launch_steps(steps)
                S.capture_logits(n + 4)
                for s, p in enumerate(prompts):
                    S.prefill(p, seq=s)
                st = binding.Stats()
                out = S.adaptive_decode(n, 0.2, cfg.exit_layers, early, st) if early else S.plain_decode(n, st)
                got.append((out, S.captured_logits()[:n].cpu().numpy()))
                assert (st.kernel_launches >= n // 2) == (steps == 1)
            assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), (n_prompt, early)
