"""Which kernels a shape's passes take (del_debug_routes, host arithmetic) against launches measured on a B200.  No GPU needed."""
import pytest

import synth
from cases import TINY

SMS = 148
MID = synth.small_variant(TINY, name="mid", d_model=1536, n_heads=24, n_kv_heads=8, head_dim=64, d_ffn=4096)
CONFIGS = dict(synth.CONFIGS, mid=MID)

# us per launch of the prefill GEMMs: tiles 256 wide, 128 wide, 128 wide with K in 2, 3, 4 parts
LAUNCHES = """
mid              48 qkv        22.4   16.1   20.0   21.0   22.5
mid              48 o          23.6   16.7   20.7   22.1   23.4
mid              48 gate_up    23.6   16.8   22.3
mid              48 down       47.6   33.0   29.0   28.1   27.9
mid             512 qkv        28.1   19.8
mid             512 o          30.4   20.1   24.7   26.1
mid             512 gate_up    26.9   30.1
mid             512 down       54.5   36.6   33.7   32.9
llama32_1b       48 qkv        26.8   19.2   21.5   22.1   23.7
llama32_1b       48 o          27.6   19.6   22.2   23.0   23.9
llama32_1b       48 gate_up    29.7   22.2
llama32_1b       48 down       83.4   57.8   41.5   35.9   34.0
llama32_1b      160 qkv        31.4   21.6   24.1   25.6
llama32_1b      160 o          33.9   22.7   25.3   26.1   27.4
llama32_1b      160 gate_up    32.0   36.8
llama32_1b      160 down       88.2   60.3   44.4   39.1   37.6
llama32_1b      512 qkv        32.5   23.2
llama32_1b      512 o          34.5   23.0   26.7
llama32_1b      512 gate_up    54.7   66.3
llama32_1b      512 down       90.2   62.4   48.1
llama32_1b     1024 qkv        33.8   36.8
llama32_1b     1024 o          34.9   24.2
llama32_1b     1024 gate_up    96.2  110.8
llama32_1b     1024 down       92.2   67.4
llama2_7b        48 qkv        49.1   35.2
llama2_7b        48 o          48.1   33.7   29.6   28.6   28.8
llama2_7b        48 gate_up    53.2   65.8
llama2_7b        48 down      112.4   78.3   51.7   43.5   40.6
llama2_7b       160 qkv        54.1   60.3
llama2_7b       160 o          53.3   35.7   33.1
llama2_7b       160 gate_up    90.4   90.8
llama2_7b       160 down      114.2   78.2   55.7
llama2_7b       512 qkv        88.9   92.2
llama2_7b       512 o          53.9   38.8
llama2_7b       512 gate_up   137.1  153.0
llama2_7b       512 down      117.9   85.0
llama2_7b      1024 qkv       141.7  187.7
llama2_7b      1024 o          59.4   70.6
llama2_7b      1024 gate_up   232.1  315.1
llama2_7b      1024 down      134.1  169.2
llama3_8b_b4    160 qkv        51.0   35.4
llama3_8b_b4    160 o          53.2   35.8   32.8
llama3_8b_b4    160 gate_up    94.5  119.1
llama3_8b_b4    160 down      144.3   99.2   66.0
llama3_8b_b4   2048 qkv       147.9  192.3
llama3_8b_b4   2048 o         105.3  133.1
llama3_8b_b4   2048 gate_up   615.3  785.9
llama3_8b_b4   2048 down      331.8  434.8
llama2_13b      160 qkv        67.0   77.6
llama2_13b      160 o          64.0   42.8
llama2_13b      160 gate_up   113.9  113.0
llama2_13b      160 down      141.5   97.5
llama2_13b     1024 qkv       223.3  272.3
llama2_13b     1024 o         118.6  122.9
llama2_13b     1024 gate_up   351.8  471.2
llama2_13b     1024 down      308.0  311.8
llama2_13b     2048 qkv       428.8  567.4
llama2_13b     2048 o         203.6  224.7
llama2_13b     2048 gate_up   732.7 1032.9
llama2_13b     2048 down      493.4  572.7
"""


@pytest.mark.parametrize("line", LAUNCHES.strip().splitlines(), ids=lambda s: "-".join(s.split()[:3]))
def test_prefill_tiles_are_near_the_best_measured(line):
    """8 %: the spread of one launch's time between runs is 2 %, the constants were fitted with 6 % rms."""
    import paper_2504_05598_b200 as dl
    name, rows, gemm, *us = line.split()
    split = dl.debug_routes(dl.make_shape(CONFIGS[name]), SMS, int(rows), int(rows))[2][["qkv", "o", "gate_up", "down"].index(gemm)]
    us = dict(zip([(256, 1), (128, 1), (128, 2), (128, 3), (128, 4)], map(float, us)))
    assert us[split] <= 1.08 * min(us.values()), (split, us)


# d_model, heads, kv heads, head dimension, d_ffn; then us per layer of a pass of so many rows: register streaming / tcgen05
PASSES = """
1536,24,8,64,4096        4:27/44 5:31/44 8:33/46 9:43/51 16:48/52 17:58/70 24:64/74 32:71/81 33:88/93 48:116/104 64:135/138
1792,28,4,64,4864        4:32/50 5:36/50 8:38/52 9:51/57 16:61/62 17:73/81 24:82/88 32:93/99 33:116/112 48:153/130 64:182/170
2048,32,8,64,4608        4:31/47 5:35/48 8:39/50 9:49/53 16:57/55 17:72/73 24:78/77 32:86/83 33:108/95 48:136/104 64:166/143
2048,32,4,64,5632        4:35/51 5:39/51 8:43/53 9:58/59 16:68/62 17:85/78 24:93/82 32:105/92 33:130/107 48:168/121 64:207/164
2048,32,8,64,8192        4:36/54 5:45/55 8:46/57 9:63/60 16:72/62 17:93/77 24:99/80 32:109/86 33:136/98 48:176/104 64:214/136
4096,32,32,128,11008     4:81/88 5:88/90 8:94/91 9:124/93 16:141/95 17:223/105 24:235/107 32:258/112 33:324/122 48:392/127 64:509/148
4096,32,8,128,14336      4:88/93 5:97/95 8:106/97 9:137/98 16:157/102 17:242/113 24:256/117 32:280/124 33:355/138 48:432/149 64:561/183
4608,36,36,128,12288     4:97/102 5:108/106 8:114/106 9:151/106 16:175/109 17:244/119 24:260/122 32:286/128 33:373/137 48:456/142 64:565/169
4864,38,38,128,13056     4:112/112 5:130/112 8:141/114 9:190/116 16:220/119 17:315/129 24:334/132 32:365/139 33:468/147 48:575/153 64:718/178
5120,40,40,128,13824     4:123/123 5:144/123 8:156/124 9:208/125 16:240/128 17:330/142 24:350/143 32:382/151 33:490/164 48:605/169 64:750/197
256,4,4,64,688           4:17/33 5:17/34 8:16/34 9:23/37 16:23/37 17:29/49 24:29/50 32:32/52 33:47/62 48:54/65 64:58/78
"""


@pytest.mark.parametrize("line", PASSES.strip().splitlines(), ids=lambda s: s.split()[0])
def test_layer_passes_are_not_slower_than_register_streaming(line):
    """3 %: the spread of a pass's time between runs."""
    import paper_2504_05598_b200 as dl
    shape, *rows = line.split()
    d, nh, nkv, hd, F = map(int, shape.split(","))
    cfg = synth.small_variant(TINY, d_model=d, n_heads=nh, n_kv_heads=nkv, head_dim=hd, d_ffn=F)
    rows_min = dl.debug_routes(dl.make_shape(cfg), SMS, 1, 1)[0]
    for r in rows:
        n, (streaming, tc) = int(r.split(":")[0]), map(float, r.split(":")[1].split("/"))
        assert n < rows_min or tc <= 1.03 * streaming, (rows_min, r)
