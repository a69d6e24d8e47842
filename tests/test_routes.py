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
