"""Decode attention where one task's key range holds more pages than a warp has lanes, and rounds whose query tiles share pages that
are copied ahead of the wait for the queries."""
import numpy as np
import pytest

import synth
from cases import TINY, TINY_GQA
from parity import ref_from_oracle, run_batch

pytestmark = pytest.mark.gpu

# 64 kv heads leave at most two key ranges per head on 148 SMs: 1 100 positions are 35 pages per range
WIDE64 = synth.small_variant(TINY, name="wide64", n_layers=2, e_max=1, d_model=256, n_heads=64, n_kv_heads=64, head_dim=64, d_ffn=272,
                             emb_scale=10.0, gain_spread=0.1, init_window=32, seed=41)
WIDE128 = synth.small_variant(WIDE64, name="wide128", n_heads=128, head_dim=128, seed=42)


@pytest.mark.parametrize("prompt_len", [1023, 1100])
@pytest.mark.parametrize("cfg", [WIDE64, WIDE128], ids=lambda c: c.name)
def test_long_key_ranges_against_prefill_kernels(cfg, prompt_len):
    """64-row passes through the decode attention against the prefill attention; the former rounds queries and probabilities to
    bf16 (2^-9 each), the latter does not: 2^-7 of a vector's norm."""
    import paper_2504_05598_b200 as dl
    cfg = synth.small_variant(cfg, prompt_len=prompt_len, gen_len=4)
    ctx = dl.DelContext(dl.make_shape(cfg), dl.upload_weights(synth.make_weights(cfg)))
    got = []
    for more in (0, dl.FLAG_NO_BULK_PREFILL):
        ctx.set_flags(dl.FLAG_PDL | dl.FLAG_TC | more)
        ctx.prefill(0, synth.make_prompt(cfg), 2)
        at = (0, 511, 512, prompt_len - 33, prompt_len - 1)
        got.append([ctx.get_hidden(0, l, j) for l in range(1, cfg.n_layers + 1) for j in (0, 15, 31)] +
                   [x for l in range(1, cfg.n_layers + 1) for pos in at for x in ctx.get_kv(0, l, pos)])
    for a, b in zip(*got):
        assert np.linalg.norm(a - b) <= 2.0 ** -7 * np.linalg.norm(a)
    ctx.close()


@pytest.mark.parametrize("batch,g_max,prompt_len", [(1, 12, 95), (3, 9, 200), (2, 4, 465)])
def test_rounds_over_committed_pages_against_oracle(batch, g_max, prompt_len):
    """Rounds on grouped queries, whose verify passes have several query tiles; the pages at the prompt's end are partly committed
    (copied early) and partly new."""
    import paper_2504_05598_b200 as dl
    cfg = synth.small_variant(TINY_GQA, batch=batch, g_max=g_max, prompt_len=prompt_len, gen_len=24)
    w = synth.make_weights(cfg)
    ctx = dl.DelContext(dl.make_shape(cfg), dl.upload_weights(w))
    refs = [ref_from_oracle(cfg, w, synth.make_prompt(cfg, s)) for s in range(batch)]
    reps = run_batch(ctx, refs, cfg.gen_len)
    for s, rep in enumerate(reps):
        assert rep.ok(), (s, rep.failures[:5])
        assert rep.rounds == len(refs[s].rounds)
    ctx.close()
