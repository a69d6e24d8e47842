"""Decode attention where one task's key range holds more pages than a warp has lanes, and rounds whose query tiles share pages that
are copied ahead of the wait for the queries."""
import functools

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
    """Rounds on grouped queries with the layer and draft length chosen per round: drafts are short here (up to 10 query rows per kv
    head, one query tile), the pages at the prompt's end partly committed and partly new."""
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


# attention makes up most of these hidden states (small embeddings), so that a page left out or taken twice shows
MANY = dict(name="many", n_layers=3, e_max=2, d_model=256, d_ffn=272, emb_scale=1.0, gain_spread=0.1, init_window=32, g_max=16, gen_len=40)


def many(hd, nkv, group):
    return synth.small_variant(TINY, **dict(MANY, head_dim=hd, n_kv_heads=nkv, n_heads=nkv * group, seed=50 + group + hd))


@functools.lru_cache(maxsize=2)
def many_weights(cfg):
    import paper_2504_05598_b200 as dl
    return dl.upload_weights(synth.make_weights(cfg))


def key_ranges(cfg, lengths, g, sms):
    """(query tiles, key ranges per head, pages of a range, committed pages of the first range) per sequence of a verify pass."""
    n_mt = -(-(g + 1) * (cfg.n_heads // cfg.n_kv_heads) // 16)
    lanes = 8 // (4 if n_mt >= 3 else n_mt)
    per_warp = -(-((max(lengths) + g + 1 + 15) // 16) // lanes)
    ns = 1 if per_warp <= 2 else max(1, min(per_warp, sms // (len(lengths) * cfg.n_kv_heads), 16))
    pages = [-(-((n + g + 1 + 15) // 16) // ns) for n in lengths]
    return n_mt, ns, pages, [min(p, n // 16) for p, n in zip(pages, lengths)]


def check_round_rows(cfg, lengths, g):
    """A round of g drafts at E = 1 on prompts of these lengths: the hidden states and cache rows of its g + 1 rows against the prefill
    kernels on the same tokens.  The decode attention rounds queries and probabilities to bf16 (2^-9 each), the prefill's does not:
    2^-7 of a vector's norm."""
    import paper_2504_05598_b200 as dl
    cfg = synth.small_variant(cfg, prompt_len=max(lengths) + 20, batch=len(lengths))
    ctx = dl.DelContext(dl.make_shape(cfg), many_weights(many(cfg.head_dim, cfg.n_kv_heads, cfg.n_heads // cfg.n_kv_heads)))
    prompts = [np.asarray(synth.make_prompt(cfg, i)[:n]) for i, n in enumerate(lengths)]
    first = [ctx.prefill(i, p, g + 2).tokens[0] for i, p in enumerate(prompts)]
    for i in range(len(lengths)):
        ctx.set_policy(i, 1, g)
    outs = ctx.round()
    L = cfg.n_layers

    def rows(i, slot0):
        n = lengths[i]
        return ([ctx.get_hidden(i, l, slot0 + k) for l in range(1, L + 1) for k in range(g + 1)] +
                [x for l in range(1, L + 1) for k in range(g + 1) for x in ctx.get_kv(i, l, n + k)])

    got = [rows(i, 0) for i in range(len(lengths))]
    fed = [np.concatenate([p, [t], ctx.get_drafts(i)[:g]]).astype(np.int32) for i, (p, t) in enumerate(zip(prompts, first))]
    assert all(o.g == g for o in outs)
    for i, tokens in enumerate(fed):
        ctx.release(i)
        ctx.prefill(i, tokens, 2)
        for a, b in zip(got[i], rows(i, cfg.init_window - (g + 1))):
            assert np.linalg.norm(a - b) <= 2.0 ** -7 * np.linalg.norm(b)
    ctx.close()


@pytest.mark.parametrize("hd,nkv,group,lengths,g,tiles,ranges", [
    (64, 64, 4, [1100], 12, 4, 2),               # two ranges of 35 pages: three chunks of 12
    (128, 64, 2, [1100], 12, 2, 2),              # six chunks of 6
    (64, 64, 4, [1550, 1200], 12, 4, 1),         # one range of 98 pages, the other sequence's 76
    (128, 64, 2, [1033, 1550], 15, 2, 1),
    (64, 64, 5, [1100, 400], 12, 5, 1),          # more than four query tiles: the pages are staged twice
    (128, 64, 5, [700, 1100], 12, 5, 1),
    (64, 64, 4, [1100], 16, 5, 2),
], ids=str)
def test_rounds_over_many_pages(hd, nkv, group, lengths, g, tiles, ranges):
    """Ranges of three and more chunks (the first two are copied before the wait, the third takes the first one's place) and of more
    pages than a warp holds ids of (32)."""
    import torch
    cfg = many(hd, nkv, group)
    n_mt, ns, pages, early = key_ranges(cfg, lengths, g, torch.cuda.get_device_properties(0).multi_processor_count)
    chunk = 12 if hd == 64 else 6
    assert (n_mt, ns) == (tiles, ranges) and max(pages) > 32 and min(early) >= 2 * chunk
    check_round_rows(cfg, lengths, g)


@pytest.mark.parametrize("hd,nkv,group,g", [(64, 80, 4, 12), (128, 80, 2, 12), (64, 80, 5, 12), (64, 2, 4, 9)], ids=str)
@pytest.mark.parametrize("length", [33, 79, 95, 96, 112, 176, 191, 192, 208, 384, 385])
def test_rounds_where_committed_pages_end(hd, nkv, group, g, length):
    """The last committed page at every place of the first two chunks of 6 or 12 (one range per head; with two kv heads ranges of one
    to a few pages)."""
    check_round_rows(many(hd, nkv, group), [length], g)
