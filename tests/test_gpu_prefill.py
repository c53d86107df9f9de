"""The dense prompt pass at the edges of its tiles, blocks and work division, against the prompt pass through the
decode kernel (eight positions at a time)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2506_03700_b200 import binding, synth


def _model(head_dim, n_q, n_kv, d_model=256, d_ff=704, layers=2):
    cfg = synth.small_config(dtype="bf16", n_layers=layers, d_model=d_model, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=head_dim,
                             d_ff=d_ff, vocab=1024, sigma=0.06, resid_scale=0.8, exit_layers=(1,))
    return cfg, binding.Model(cfg, synth.make_weights(cfg, device="cuda"))


def _compare(cfg, gm, n, page_tokens=64):
    prompt = synth.make_prompt(cfg, n=n).numpy()
    out = []
    for dense in (True, False):
        S = binding.Session(gm, 1, n + 40, page_tokens if dense else 64, 0)
        S.capture_logits(4)
        S.set_prefill(dense)
        S.prefill(prompt)
        pos = sorted({p for p in (0, 1, 31, 63, 64, 127, 128, 129, 255, 256, n // 2, n - 2, n - 1) if 0 <= p < n})
        kv = np.stack([S.read_kv(w, l, p) for l in range(cfg.n_layers) for p in pos for w in (0, 1)])
        out.append((S.state(), kv, S.captured_logits().cpu().numpy()))
    (sd, kd, ld), (sc, kc, lc) = out
    assert sd[0] == sc[0] == n + 1 and np.array_equal(sd[1], sc[1])
    # Both sides hold fp32 sums of the same bf16 products; they differ where a sum's last bits decide the cache's bf16
    # rounding (one step is at most 2^-7 of a value, i.e. below 2^-8 of the largest of a row twice its size), and by what
    # such steps move in the layer above.
    assert np.abs(kd - kc).max() <= 2.0 ** -7 * np.abs(kc).max() * 1.5
    assert np.linalg.norm(kd - kc) <= 1e-3 * np.linalg.norm(kc)
    assert np.linalg.norm(ld[0] - lc[0]) <= 5e-3 * np.linalg.norm(lc[0])


@pytest.mark.parametrize("n", [9, 31, 32, 33, 64, 65, 128, 129, 256, 257, 513, 800])
def test_tile_edges(n):
    _compare(*_model(64, 4, 2), n)


@pytest.mark.parametrize("hd,nq,nkv,d,dff", [(128, 4, 1, 512, 1088), (128, 3, 3, 320, 64), (64, 5, 5, 64, 192), (64, 12, 3, 1152, 2624)])
def test_shapes_of_the_fused_epilogues(hd, nq, nkv, d, dff):
    """Widths that are no multiples of a tile, of a head pair or of an accumulator chunk."""
    _compare(*_model(hd, nq, nkv, d, dff), 150)


@pytest.mark.parametrize("n", [2048, 2049, 4100])
def test_block_edges(n):
    _compare(*_model(64, 4, 1), n)


@pytest.mark.parametrize("page_tokens", [16, 32, 128, 256])
def test_page_sizes(page_tokens):
    _compare(*_model(128, 2, 1), 300, page_tokens)


def test_separate_and_fused_tensors_give_the_same_cache():
    """q, k, v and gate, up lent as separate tensors go through the same tiles as slices of one."""
    cfg, gm = _model(64, 4, 2)
    w = synth.make_weights(cfg, device="cuda")
    qd, kvd = cfg.n_q_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim
    sep = {}
    for k, t in w.items():
        p = k.rsplit(".", 1)[0] + "."
        if k.endswith("wqkv"):
            for name, a, b in (("wq", 0, qd), ("wk", qd, qd + kvd), ("wv", qd + kvd, qd + 2 * kvd)):
                sep[p + name] = t[a:b].clone()
        elif k.endswith("w_gate_up"):
            sep[p + "w_gate"], sep[p + "w_up"] = t[:cfg.d_ff].clone(), t[cfg.d_ff:].clone()
        else:
            sep[k] = t
    prompt = synth.make_prompt(cfg, n=200).numpy()
    rows = []
    for m in (gm, binding.Model(cfg, sep)):
        S = binding.Session(m, 1, 256, 64, 0)
        S.prefill(prompt)
        rows.append(np.stack([S.read_kv(wh, l, p) for wh in (0, 1) for l in range(cfg.n_layers) for p in (0, 100, 199)]))
    assert np.array_equal(rows[0], rows[1])


def test_three_q_heads_per_kv_head_keep_the_decode_path():
    """The dense pass has no form for them: prompts below 32 tokens are accepted, longer ones refused, as before."""
    cfg, gm = _model(64, 6, 2)
    S = binding.Session(gm, 1, 128, 64, 0)
    S.prefill(synth.make_prompt(cfg, n=20).numpy())
    assert S.state()[0] == 21
    with pytest.raises(binding.AdaError) as e:
        S.prefill(synth.make_prompt(cfg, n=40).numpy())
    assert e.value.code == -6


def _rows(S, cfg, positions):
    return np.stack([S.read_kv(w, l, p) for l in range(cfg.n_layers) for p in positions for w in (0, 1)])


@pytest.mark.parametrize("hd,nq,nkv,d,dff", [(64, 16, 4, 1024, 3072), (128, 16, 16, 2048, 5504)])
def test_a_prefix_leaves_the_same_cache_bits_whatever_follows_it(hd, nq, nkv, d, dff):
    """The order of every sum is that of the shapes, not of the prompt's length: prompts that start alike leave the same K
    and V rows for what they share, whichever tiles, pieces and blocks the products were divided into."""
    cfg, gm = _model(hd, nq, nkv, d, dff, layers=3)
    prompt = synth.make_prompt(cfg, n=4200).numpy()
    S = binding.Session(gm, 1, 4300, 64, 0)
    seen = {}
    for n in (9, 33, 70, 140, 257, 300, 520, 777, 1024, 1500, 2048, 2049, 4200):
        S.prefill(prompt[:n])
        for p in (0, 5, 8, 32, 60, 69, 128, 139, 256, 299, 500, 519, 776, 1023, 1400, 2047, 2048):
            if p < n:
                rows = _rows(S, cfg, [p])
                first = seen.setdefault(p, (n, rows))
                assert np.array_equal(first[1], rows), (p, first[0], n)


@pytest.mark.parametrize("hd,nq,nkv,d", [(64, 16, 4, 1024), (128, 16, 16, 2048)])
@pytest.mark.parametrize("n", [9, 31, 100])
def test_first_layer_rounds_what_the_embeddings_give(hd, nq, nkv, d, n):
    """The first layer's input is bf16: its products can be as exact as their sums, whether eight positions or the whole prompt
    are multiplied at once.  A K or V differs from the rounded float64 one where an error e of the sums straddles a rounding
    boundary, i.e. with probability e / ulp: below 1.2e-6 / 2^-8 = 3e-4 (values near zero have wider errors relative to them
    than the sums' 2-norm says: twice that).  A normalised row would be split with an error of 2.5e-6 instead: 3e-3 measured."""
    cfg, gm = _model(hd, nq, nkv, d, 1024, layers=1)
    w = synth.make_weights(cfg, device="cuda")
    prompt = synth.make_prompt(cfg, n=n)
    S = binding.Session(gm, 1, n + 8, 64, 0)
    S.prefill(prompt.numpy())
    x = w["tok_embed"][prompt.long().cuda()].double()
    qkv = (x / torch.sqrt((x * x).mean(-1, keepdim=True) + np.float32(cfg.rms_eps).item())) @ w["layers.0.wqkv"].double().T
    k, v = qkv[:, nq * hd:].view(n, 2, nkv, hd).unbind(1)
    angle = torch.arange(n, dtype=torch.float64, device="cuda")[:, None] * cfg.rope_base ** (-2.0 * torch.arange(hd // 2, dtype=torch.float64, device="cuda") / hd)
    co, si = angle.cos()[:, None], angle.sin()[:, None]
    a, b = k[..., :hd // 2], k[..., hd // 2:]
    k = torch.cat([a * co - b * si, b * co + a * si], -1)
    want = torch.stack([k, v], 1).float().bfloat16().float().cpu().numpy().reshape(n, 2, nkv * hd)
    got = _rows(S, cfg, range(n)).reshape(n, 2, nkv * hd)
    assert np.mean(got != want) <= 6e-4


@pytest.mark.parametrize("hd,nq,nkv", [(64, 4, 1), (128, 4, 2), (128, 2, 2)])
@pytest.mark.parametrize("bad", ["nan", "infinity", "one value"])
@pytest.mark.parametrize("n,at", [(40, 20), (129, 127), (200, 128), (700, 513), (2100, 1060)])
def test_a_token_that_is_not_finite_leaves_the_positions_before_it_alone(hd, nq, nkv, bad, n, at):
    """Causality with values that no multiplication by zero can hide: the positions before such a token keep, bit for bit, the
    cache rows that they have without it; what follows is not finite.  "one value": a single feature of the token's value row
    of one head overflows, everything else about the token is finite."""
    cfg, _ = _model(hd, nq, nkv)
    w = synth.make_weights(cfg, device="cuda")
    w["tok_embed"][:, 3] = 0.0
    prompt = synth.make_prompt(cfg, n=n).numpy()
    token = next(t for t in range(cfg.vocab) if t not in prompt)
    prompt[at] = token
    w["tok_embed"][token, 3] = 0.5
    rows = []
    for broken in (False, True):
        if broken and bad == "one value":
            w["layers.0.wqkv"][(cfg.n_q_heads + cfg.n_kv_heads) * hd + 5, 3] = 3e38
        elif broken:
            w["tok_embed"][token, 3] = float("nan") if bad == "nan" else float("inf")
        S = binding.Session(binding.Model(cfg, w), 1, n + 8, 64, 0)
        S.prefill(prompt)
        rows.append((_rows(S, cfg, range(max(0, at - 200), at)), _rows(S, cfg, [at]), _rows(S, cfg, [n - 1])))
    (good, good_own, good_after), (before, own, after) = rows
    assert np.isfinite(good).all() and np.isfinite(good_own).all() and np.isfinite(good_after).all()
    assert np.array_equal(good, before)
    assert np.array_equal(good_after[:2], after[:2]) and np.isnan(after[2:]).all()   # layer 0 sees the token itself only, the next one all
    if bad == "one value":
        assert np.array_equal(good_own[0], own[0]) and np.flatnonzero(~np.isfinite(own[1])).tolist() == [5]
    else:
        assert np.isnan(own).all()


@pytest.mark.parametrize("hd,nq,nkv", [(64, 4, 2), (128, 2, 2)])
def test_a_wait_that_runs_out_ends_the_prompt_pass_with_a_timeout_and_the_session_recovers(hd, nq, nkv):
    """The dense pass's waits end at the session's limit like the decode kernel's: set far below what a copy takes, the call
    returns ADA_ETIMEOUT, and with the usual limit the same session gives what a fresh one gives."""
    cfg, gm = _model(hd, nq, nkv)
    prompt = synth.make_prompt(cfg, n=300).numpy()
    F = binding.Session(gm, 1, 400, 64, 0)
    F.prefill(prompt)
    S = binding.Session(gm, 1, 400, 64, 0)
    S.set_wait_limit(20)                  # nanoseconds
    with pytest.raises(binding.AdaError) as e:
        S.prefill(prompt)
    assert e.value.code == -5
    torch.cuda.synchronize()              # the context is intact
    S.set_wait_limit(2_000_000_000)
    S.reset()
    S.prefill(prompt)
    positions = (0, 127, 128, 299)
    assert np.array_equal(_rows(S, cfg, positions), _rows(F, cfg, positions))
    assert np.array_equal(S.plain_decode(4), F.plain_decode(4))
