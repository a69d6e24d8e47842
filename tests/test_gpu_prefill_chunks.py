"""Prompts in several chunks: contexts whose workspace holds fewer positions than the prompt has."""
import ctypes as C

import numpy as np
import pytest

import synth
from cases import TINY_HD128_GQA, TINY_LONG2, TINY_LONG3
from parity import ref_from_oracle, run_sequence

pytestmark = pytest.mark.gpu

# the window straddles a chunk boundary (512), tcgen05 attention
HD128_GQA_530 = synth.small_variant(TINY_HD128_GQA, name="tiny_hd128_gqa_530", prompt_len=530, seed=23)


def workspace_bytes(cfg, rows):
    """Bytes with chunk buffers of `rows` positions: fp32 H and two lists of sums of squares, two pairs of d, two of heads, one of F."""
    import paper_2504_05598_b200 as dl
    shape = dl.make_shape(cfg)
    full_rows = min(2048, (shape.max_seq + 127) // 128 * 128)
    per_row = 4 * cfg.d_model + 2 * 4 * ((cfg.d_model + 63) // 64) + 2 * 4 * cfg.d_model + 2 * 4 * cfg.n_heads * cfg.head_dim + 4 * cfg.d_ffn
    return dl.load_library().del_workspace_bytes(C.byref(shape)) - (full_rows - rows) * per_row


@pytest.mark.parametrize("rows", [128, 512])
@pytest.mark.parametrize("cfg", [TINY_LONG2, TINY_LONG3, TINY_HD128_GQA, HD128_GQA_530], ids=lambda c: c.name)
def test_chunks_against_oracle(cfg, rows):
    """Cache, the window's hidden states and the rounds that follow, as with the whole prompt in one chunk."""
    import oracle
    import paper_2504_05598_b200 as dl
    w = synth.make_weights(cfg)
    dev = dl.upload_weights(w)
    prompt = synth.make_prompt(cfg)
    P, W, L = len(prompt), cfg.init_window, cfg.n_layers
    launches = []
    for ws in (None, workspace_bytes(cfg, rows)):
        ctx = dl.DelContext(dl.make_shape(cfg), dev, workspace_bytes=ws)
        ctx.prefill(0, prompt, cfg.gen_len)
        launches.append(ctx.launch_count())
    n_chunks = -(-P // rows)
    assert launches[1] - launches[0] >= (n_chunks - 1) * (5 * L - 4)      # of the last layer a chunk before the window needs QKV alone
    o = oracle.OracleSeq(cfg, w)
    o.prefill(prompt)
    for l in range(1, L + 1):
        for pos in sorted({0, 1, 127, 128, 129, 255, 256, 383, 384, 511, 512, 513, P - W - 1, P - W, P - 1}):
            k, v = ctx.get_kv(0, l, pos)
            kr, vr = o.k_row(l, pos), o.v_row(l, pos)
            assert np.abs(k - kr).max() <= 2e-2 * np.abs(kr).max() + 1e-6, ("k", l, pos)
            assert np.abs(v - vr).max() <= 2e-2 * np.abs(vr).max() + 1e-6, ("v", l, pos)
    for l in range(L + 1):
        for j in range(W):
            r, got = o.hidden(l, j), ctx.get_hidden(0, l, j)
            assert np.abs(got - r).max() <= 2e-2 * np.abs(r).max() + 1e-6, ("h", l, j)
    o.close()
    rep = run_sequence(ctx, 0, ref_from_oracle(cfg, w, prompt), cfg.gen_len)
    assert rep.ok(), rep.failures[:5]
    ctx.close()


def test_smallest_workspace():
    """One tile of 128 positions is accepted, a byte less is not."""
    import paper_2504_05598_b200 as dl
    cfg = TINY_LONG2
    dev = dl.upload_weights(synth.make_weights(cfg))
    ctx = dl.DelContext(dl.make_shape(cfg), dev, workspace_bytes=workspace_bytes(cfg, 128))
    assert ctx.workspace_bytes == workspace_bytes(cfg, 128)
    ctx.close()
    with pytest.raises(dl.DelError) as e:
        dl.DelContext(dl.make_shape(cfg), dev, workspace_bytes=workspace_bytes(cfg, 128) - 1)
    assert e.value.code == dl.ENOSPC
