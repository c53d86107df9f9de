"""The fp32 one-launch path (host arithmetic, no GPU): which sessions take it, and that no CTA of its grid can fall so far behind
that what it has yet to read is written again.  Values pass between the CTAs without a barrier; a CTA that owns an output between
its read of a buffer and the next writing of that buffer holds the writers back, because they wait for that output."""

import ctypes

import pytest

from paper_2506_03700_b200 import binding, synth

# phases of a layer, in order; for every buffer that all CTAs read: the phase that reads it and the phase, a layer later, that
# writes it again.  (Queries, keys and values are read by CTAs with an attention item only, which publish that item's result in the
# same phase; the attention phase itself, whose items depend on the positions, counts for nobody.)
PHASES = ["qkv", "attention", "o", "gate_up", "down"]
BUFFERS = {"XA": ("qkv", "down"), "XB": ("gate_up", "o"), "HT": ("down", "gate_up"), "PT": ("o", "attention")}


@pytest.mark.parametrize("sms", [1, 132, 148, 160, 300])
@pytest.mark.parametrize("shape", [(1, 1, 32, 8, 8), (1, 1, 32, 64, 128), (2, 1, 32, 128, 64), (4, 2, 32, 128, 344), (6, 2, 32, 144, 2048),
                                   (2, 2, 32, 152, 8), (4, 4, 64, 256, 688), (2, 1, 128, 512, 136), (16, 4, 64, 1024, 2816), (32, 8, 64, 2048, 5632)])
def test_every_cta_holds_back_the_writers_of_what_it_reads(shape, sms):
    nq, nkv, hd, d, dff = shape
    cfg = synth.small_config(n_layers=2, d_model=d, n_q_heads=nq, n_kv_heads=nkv, head_dim=hd, d_ff=dff, vocab=100)
    plans = [binding.debug_resident_plan(cfg, 1, 5, sms, c) for c in range(sms + 1)]
    grid = plans[0]["grid"]
    assert 1 <= grid <= sms
    want = dict(qkv=(nq + 2 * nkv) * hd // 2, o=d, gate_up=dff, down=d)
    for ph, n in want.items():
        assert sum(p[ph] for p in plans) == n and all(p[ph] == 0 for p in plans[grid:]), ph
    for c, p in enumerate(plans[:grid]):
        for buf, (reader, writer) in BUFFERS.items():
            r, w = PHASES.index(reader), PHASES.index(writer)
            between = [PHASES[i % 5] for i in range(r, w if w > r else w + 5)]
            assert any(p.get(ph, 0) > 0 for ph in between), (c, buf)
        # head partials and staged logits are read behind a head and written again by the next one: a layer at least lies between
        assert any(p[ph] > 0 for ph in want), c


# (width, layers, d_ff, vocabulary, sequences, early tokens): decode calls in one launch, prompts in one launch.  Both sides of every
# line of the rule, as they were measured (the ratios stand beside the rule).
ROUTES = [((256, 4, 688, 2048, 1, 5), True, True), ((256, 4, 688, 2048, 8, 5), True, True), ((256, 4, 688, 2048, 16, 0), True, True),
          ((64, 4, 176, 2048, 16, 3), True, True), ((320, 4, 896, 2048, 12, 1), True, False), ((256, 4, 688, 8192, 8, 0), True, False),
          ((256, 4, 688, 32000, 8, 0), False, False), ((256, 4, 688, 32000, 3, 5), True, False), ((256, 4, 688, 64000, 1, 5), False, False),
          ((256, 12, 688, 64000, 1, 5), True, False), ((384, 4, 1024, 2048, 3, 5), True, False), ((384, 4, 1024, 2048, 8, 0), False, False),
          ((512, 4, 1408, 8192, 2, 5), True, False), ((512, 4, 1408, 8192, 3, 1), False, False), ((512, 4, 1408, 32000, 1, 5), False, False),
          ((1024, 24, 2816, 32000, 1, 5), True, False), ((1024, 24, 2816, 32000, 4, 1), False, False), ((1024, 4, 2816, 32000, 1, 5), False, False),
          ((2048, 16, 5632, 32000, 1, 5), False, False),
          ((256, 4, 688, 2048, 1, 16), False, False), ((256, 4, 688, 2048, 16, 3), False, False)]   # (the kernel's tables; shared memory)


@pytest.mark.parametrize("shape,decode,prompts", ROUTES)
def test_sessions_take_the_path_that_measured_faster(shape, decode, prompts):
    d, n_layers, dff, vocab, batch, max_early = shape
    hd = 64 if d >= 256 else 32
    cfg = synth.small_config(n_layers=n_layers, d_model=d, n_q_heads=d // hd, n_kv_heads=1, head_dim=hd, d_ff=dff, vocab=vocab)
    p = binding.debug_resident_plan(cfg, batch, max_early)
    assert (p["rows"] > 0, bool(p["prompts"])) == (decode, prompts)
    if decode:
        assert p["rows"] >= batch * (max_early + 1)
    bf16 = synth.small_config(n_layers=n_layers, d_model=d, n_q_heads=d // hd, n_kv_heads=1, head_dim=hd, d_ff=dff, vocab=vocab, dtype="bf16")
    assert binding.debug_resident_plan(bf16, batch, max_early)["rows"] == 0


def test_sessions_that_do_not_take_it_reserve_nothing_for_it():
    """Scratch of a wide fp32 session: no exchanged words (8192 positions: 8 rows x 32 heads x 64 chunks x 130 words of 8 bytes alone
    would be 17 MB), as for the same session with room for more early tokens than the kernel's tables hold."""
    lib = binding.load()
    h = ctypes.c_void_p()
    cfg = binding.Config(16, 4096, 32, 8, 128, 11008, 32000, 0, 1, 10000.0, 1e-5)
    assert lib.ada_model_create(ctypes.byref(cfg), ctypes.byref(h)) == 0
    # up to 32 rows the buffers of the per-operation path do not depend on max_early
    assert lib.ada_session_scratch_bytes(h, 1, 8192, 5) == lib.ada_session_scratch_bytes(h, 1, 8192, 16)
    lib.ada_model_destroy(h)
