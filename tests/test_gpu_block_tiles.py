"""The one-launch kernel on bulk copies (float32 layers): sizes at which its tiles, blocks of weights and copies have remainders.

Rows that start between 16-byte boundaries (input and output widths that are no multiple of 4), one to four tokens per warp in the
descent and more than one round of it, tiles of 8, 16 and 32 tokens, leaves whose weights take one block and several, fewer than
eight units in the last block, one to four outputs per thread; next to widths that do not fit it.  The same bits as a warp per
token (the sums are added in the same order)."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
CASES = [
    C("bt_d3_narrow", 784, 10, 3, 32, "relu", "f32", 2048, "normal"),
    C("bt_one_leaf", 5, 3, 0, 1, "gelu", "f32", 700, "normal"),
    C("bt_d1", 33, 1, 1, 4, "gelu", "f32", 2501, "normal", node_bias_std=0.3),
    C("bt_d2_ragged", 253, 39, 2, 13, "silu", "f32", 5003, "normal"),
    C("bt_d6_three_tokens", 130, 257, 6, 9, "gelu", "f32", 6304, "normal"),
    C("bt_d8_three_outputs", 768, 768, 8, 12, "gelu", "f32", 3000, "layernorm"),
    C("bt_d4_wide", 1024, 1024, 4, 33, "gelu_tanh", "f32", 1500, "normal"),
    C("bt_d4_ragged_wide", 1021, 1023, 4, 20, "gelu", "f32", 1300, "normal"),
    C("bt_d5_many", 64, 48, 5, 16, "relu", "f32", 20011, "clusters"),
    C("bt_d9_empty_leaves", 72, 520, 9, 12, "gelu", "f32", 6000, "clusters"),
    C("bt_d3_long_rows", 1300, 40, 3, 8, "gelu", "f32", 900, "normal"),
    C("bt_d3_too_long", 2056, 40, 3, 8, "gelu", "f32", 900, "normal"),
    C("bt_d2_too_many_outputs", 64, 1100, 2, 8, "gelu", "f32", 900, "normal"),
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_block_tiles_match_the_oracle(cfg):
    case = util.make_case(cfg, seed=9)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "f32")
    for _ in range(2):
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_launch_count() == 1 and layer.last_status() == 0
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        util.check_outputs(y, y_ref, "f32")
    layer.set_path("warp")
    y2, leaf2 = layer.forward_infer(x)
    assert torch.equal(y2, y) and torch.equal(leaf2, leaf)
    layer.close()
