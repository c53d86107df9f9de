"""Several sequences with several early tokens each on one weight stream: the persistent kernel of 24 token columns against the
same sequences decoded alone by the kernel of eight, bit for bit."""

import numpy as np
import pytest
import torch

from paper_2506_03700_b200 import binding, synth

pytestmark = pytest.mark.gpu

LENS = [5, 131, 70, 33, 8, 127, 12, 260]
TAPE = [1, 1, 0, 1, 2, 1, 1, 1, 0, 0, 1, 2, 1] * 12


def model(heads, kv, hd, **kw):
    cfg = synth.small_config(dtype="bf16", n_layers=4, d_model=256, n_q_heads=heads, n_kv_heads=kv, head_dim=hd, sigma=0.08, resid_scale=0.8,
                             exit_layers=(1, 2), **kw)
    gm = binding.Model(cfg, synth.make_weights(cfg, device="cuda", norm_gain_jitter=0.1))
    gm.set_exit_head(1, None, 4.0)
    gm.set_exit_head(2, synth.make_head_transform(cfg, 2, device="cuda", noise=0.1), 4.0)
    return cfg, gm


def run(gm, cfg, prompts, n, max_early, mode, tape):
    S = binding.Session(gm, len(prompts), 320, 64, max_early)
    assert S.get_path() == 1
    S.capture_logits(n)
    for i, p in enumerate(prompts):
        S.prefill(p, seq=i)
    st = binding.Stats()
    if mode == "plain":
        out = S.plain_decode(n, st)
    else:
        if tape:
            S.set_exit_tape(TAPE)   # sequence 0 leaves against its heads' decisions: rejected tokens, rolled back caches
        # the first half accepts every early prediction it may make, the second decides by the heads
        out = np.concatenate([S.adaptive_decode(n // 2, 0.0, cfg.exit_layers, max_early, st),
                              S.adaptive_decode(n - n // 2, 0.3, cfg.exit_layers, max_early, st)], axis=1)
        assert st.early_exits > 0
    return out, S.captured_logits().clone(), st


# sequences x (early tokens + 1): two and three column tiles in use, all 24 columns, groups with a remainder, eight sequences
@pytest.mark.parametrize("max_early,batch", [(5, 2), (5, 4), (4, 5), (7, 3), (2, 8), (5, 5)])
@pytest.mark.parametrize("shape", [(4, 1, 64), (4, 4, 128), (6, 2, 64)])
@pytest.mark.parametrize("mode", ["plain", "adaptive"])
def test_sequences_equal_their_own_runs(max_early, batch, shape, mode):
    # (d_ff and vocabulary that the tiles of sixteen rows and the chunks of 512 do not divide evenly over the CTAs)
    cfg, gm = model(*shape, d_ff=1088 if shape[2] == 128 else 704, vocab=5000 if shape[0] == 6 else 2048)
    # (three q heads per kv head: prompts of 32 tokens and more are refused)
    prompts = [synth.make_prompt(cfg, n=min(k, 31) if shape[0] == 6 else k, seq=i).numpy() for i, k in enumerate(LENS[:batch])]
    n = 22
    out, lg, st = run(gm, cfg, prompts, n, max_early, mode, True)
    one, lg1, s1 = run(gm, cfg, prompts[:1], n, max_early, mode, True)
    assert np.array_equal(out[0], one[0]) and torch.equal(lg, lg1)
    for i in range(1, batch):
        alone, _, _ = run(gm, cfg, prompts[i:i + 1], n, max_early, mode, False)
        assert np.array_equal(out[i], alone[0]), i
    if mode == "plain":   # one pass of the weights per step for every group that 24 columns hold
        groups = -(-batch // min(8, 24 // (max_early + 1)))
        assert st.layer_passes == groups * s1.layer_passes


def test_wide_products_of_the_13b_layer():
    """Two layers of the 13B shape (forty kv heads, products cut unevenly over the CTAs, more attention items than CTAs, elements
    past the stash): four sequences with five early tokens equal their own runs."""
    cfg = synth.small_config(dtype="bf16", n_layers=2, d_model=5120, n_q_heads=40, n_kv_heads=40, head_dim=128, d_ff=13824, vocab=32000,
                             sigma=0.02, resid_scale=0.2, exit_layers=(1,))
    gen = torch.Generator(device="cuda").manual_seed(3)
    nrm = lambda *s: torch.empty(*s, dtype=torch.bfloat16, device="cuda").normal_(0, 0.02, generator=gen)
    one = torch.ones(cfg.d_model, dtype=torch.bfloat16, device="cuda")
    w = {"tok_embed": nrm(cfg.vocab, cfg.d_model), "final_norm": one}
    for l in range(2):
        p = "layers.%d." % l
        w[p + "attn_norm"] = w[p + "ffn_norm"] = one
        w[p + "wqkv"], w[p + "wo"] = nrm(cfg.qkv_rows, cfg.d_model), nrm(cfg.d_model, cfg.d_model)
        w[p + "w_gate_up"], w[p + "w_down"] = nrm(2 * cfg.d_ff, cfg.d_model), nrm(cfg.d_model, cfg.d_ff)
    gm = binding.Model(cfg, w)
    gm.set_exit_head(1, None, 1.0)
    prompts = [synth.make_prompt(cfg, n=k, seq=i).numpy() for i, k in enumerate((150, 290, 33, 200))]
    outs = []
    for ps in [prompts] + [[p] for p in prompts]:
        S = binding.Session(gm, len(ps), 320, 64, 5)
        for i, p in enumerate(ps):
            S.prefill(p, seq=i)
        outs.append(S.adaptive_decode(14, 0.0, cfg.exit_layers, 5))
    for i in range(4):
        assert np.array_equal(outs[0][i], outs[1 + i][0]), i
