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
        for how in ("plain", "adaptive", "per-operation"):
            S = binding.Session(gm, 1, 768, 64, 5)
            S.set_prefill(False)
            S.capture_logits(n + 4)
            S.prefill(prompt)
            if how == "per-operation":
                S.set_path(0)
            out = S.adaptive_decode(n, 0.0, cfg.exit_layers, 5) if how == "adaptive" else S.plain_decode(n)
            got.append((out[0], S.captured_logits()[:n].cpu().numpy()))
        (tp, lp), (ta, la), (to, lo) = got
        # every token leaves early (threshold 0), up to six columns in flight: the same bits as one column at a time
        assert np.array_equal(tp, ta) and np.array_equal(lp, la), n_prompt
        # the per-operation kernels share the cache of the prompt; what they add to it differs by bf16 roundings of K and V
        # (2^-9 of a value each) in at most n of the positions
        same = int(np.argmin(np.append(tp == to, False)))
        assert same >= 1 and np.linalg.norm(lp[:same] - lo[:same]) <= 5e-3 * np.linalg.norm(lo[:same]), n_prompt
