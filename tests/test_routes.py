"""Which kernels a shape's passes take (del_debug_routes, host arithmetic) against launches measured on a B200.  No GPU needed."""
import pytest

import synth
from cases import TINY

SMS = 148
MID = synth.small_variant(TINY, name="mid", d_model=1536, n_heads=24, n_kv_heads=8, head_dim=64, d_ffn=4096)
CONFIGS = dict(synth.CONFIGS, mid=MID)

# us per launch of the prefill GEMMs: tiles 256 wide, 128 wide, 128 wide with K in 2, 3, 4 parts
LAUNCHES = """
mid              48 qkv        22.7   16.4   20.0   21.1   22.7
mid              48 o          23.9   16.8   20.6   21.9   23.0
mid              48 gate_up    23.3   17.0   22.0
mid              48 down       48.2   33.4   29.4   28.3   28.0
mid             512 qkv        28.2   19.9
mid             512 o          30.2   20.2   24.6   26.0
mid             512 gate_up    26.6   29.9
mid             512 down       54.0   36.5   33.4   32.5
llama32_1b       48 qkv        30.1   20.7   23.1   23.9   24.9
llama32_1b       48 o          30.4   20.6   23.6   24.1   24.7
llama32_1b       48 gate_up    32.2   23.2
llama32_1b       48 down       92.5   61.4   44.5   38.5   35.7
llama32_1b      160 qkv        32.0   22.3   25.1   26.0
llama32_1b      160 o          33.9   22.8   25.8   26.4   27.7
llama32_1b      160 gate_up    32.4   37.5
llama32_1b      160 down       89.6   60.8   45.2   40.1   38.3
llama32_1b      512 qkv        32.6   23.2
llama32_1b      512 o          34.1   23.1   26.5
llama32_1b      512 gate_up    54.8   66.8
llama32_1b      512 down       90.8   63.0   47.7
llama32_1b     1024 qkv        33.8   36.8
llama32_1b     1024 o          34.9   24.2
llama32_1b     1024 gate_up    96.2  110.8
llama32_1b     1024 down       92.2   67.4
llama2_7b        48 qkv        49.5   35.2
llama2_7b        48 o          49.0   33.5   30.1   29.0   29.3
llama2_7b        48 gate_up    53.0   63.7
llama2_7b        48 down      112.9   76.9   52.5   44.4   41.5
llama2_7b       160 qkv        55.3   61.1
llama2_7b       160 o          53.3   36.1   33.7
llama2_7b       160 gate_up    91.5   90.3
llama2_7b       160 down      115.4   79.3   56.6
llama2_7b       512 qkv        88.8   92.2
llama2_7b       512 o          53.8   39.2
llama2_7b       512 gate_up   136.8  153.8
llama2_7b       512 down      117.9   87.2
llama2_7b      1024 qkv       141.7  187.7
llama2_7b      1024 o          59.4   70.6
llama2_7b      1024 gate_up   232.1  315.1
llama2_7b      1024 down      134.1  169.2
llama3_8b_b4    160 qkv        51.4   36.2
llama3_8b_b4    160 o          53.8   36.4   33.6
llama3_8b_b4    160 gate_up    95.0  118.9
llama3_8b_b4    160 down      145.0   99.2   67.0
llama3_8b_b4   2048 qkv       147.9  192.3
llama3_8b_b4   2048 o         105.3  133.1
llama3_8b_b4   2048 gate_up   615.3  785.9
llama3_8b_b4   2048 down      331.8  434.8
llama2_13b      160 qkv        67.7   75.6
llama2_13b      160 o          64.5   43.5
llama2_13b      160 gate_up   114.7  112.4
llama2_13b      160 down      142.4   97.8
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
1536,24,8,64,4096        4:28/46 5:32/45 8:34/47 9:45/52 16:50/53 17:59/71 24:66/76 32:72/81 33:91/93 48:119/104 64:137/140
1792,28,4,64,4864        4:32/51 5:37/51 8:39/53 9:52/59 16:62/63 17:75/82 24:83/87 32:94/100 33:118/112 48:157/129 64:186/172
2048,32,8,64,4608        4:32/50 5:37/51 8:40/53 9:52/56 16:58/58 17:75/76 24:79/81 32:87/86 33:112/98 48:140/107 64:168/144
2048,32,4,64,5632        4:34/53 5:40/53 8:43/55 9:59/61 16:69/65 17:86/82 24:93/84 32:105/93 33:133/109 48:171/122 64:208/165
2048,32,8,64,8192        4:36/59 5:44/58 8:47/60 9:64/64 16:73/64 17:94/81 24:100/85 32:110/90 33:141/103 48:180/111 64:216/145
4096,32,32,128,11008     4:83/96 5:89/95 8:93/98 9:126/102 16:141/102 17:224/116 24:236/118 32:258/124 33:327/137 48:393/141 64:508/162
4096,32,8,128,14336      4:88/103 5:99/101 8:106/104 9:138/105 16:158/110 17:245/124 24:256/126 32:280/132 33:359/148 48:432/156 64:561/187
4608,36,36,128,12288     4:99/111 5:105/111 8:115/113 9:149/117 16:171/118 17:244/132 24:262/134 32:285/139 33:372/152 48:450/155 64:564/173
4864,38,38,128,13056     4:116/121 5:130/122 8:137/123 9:189/131 16:214/130 17:315/142 24:332/145 32:361/148 33:470/165 48:573/170 64:715/187
5120,40,40,128,13824     4:126/131 5:140/132 8:148/132 9:205/138 16:234/139 17:329/154 24:348/155 32:378/161 33:493/176 48:606/179 64:746/201
256,4,4,64,688           4:18/33 5:17/33 8:17/34 9:23/36 16:24/36 17:30/50 24:31/50 32:33/52 33:49/63 48:54/66 64:58/79
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
