"""The grid of the fp32 one-launch path (host arithmetic, no GPU): no CTA can fall so far behind that what it has yet to read is
written again.  Values pass between the CTAs without a barrier; a CTA that owns an output between its read of a buffer and the
next writing of that buffer holds the writers back, because they wait for that output."""

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
    plans = [binding.debug_resident_plan(cfg, sms, c) for c in range(sms + 1)]
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
