"""Leaf kernel with a warp per tile of up to 16 tokens (thin buckets of many leaves) against the oracle: widths that are no
multiple of its 32-column and 32-output blocks, leaves with none, a few, 16 and many more tokens, every hidden width it takes."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
CASES = [
    C("wt_d9_l8", 128, 64, 9, 8, "gelu", "bf16", 4500, "normal"),
    C("wt_d9_ragged", 328, 272, 9, 13, "silu", "bf16", 5001, "clusters"),            # 41 units of 8 columns, 8.5 blocks of outputs
    C("wt_d10_padded", 200, 48, 10, 16, "relu", "bf16", 2500, "normal", node_bias_std=0.3),
    C("wt_d11_thin", 256, 256, 11, 10, "gelu", "bf16", 4097, "normal"),
    C("wt_d9_full_tiles", 64, 32, 9, 16, "gelu_tanh", "bf16", 20000, "clusters"),    # leaves of hundreds of tokens beside empty ones
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_warp_tiles_match_the_oracle(cfg):
    case = util.make_case(cfg, seed=9)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, cfg.dtype)
    layer.profile_begin(1)
    y_first = None
    for _ in range(2):                                     # the second call starts from the counts the first one cleared
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_status() == 0
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        util.check_outputs(y, y_ref, cfg.dtype)
        assert y_first is None or torch.equal(y, y_first)  # whatever the order of the lists was
        y_first = y
    names = [n for n, _ in layer.profile_end()[0]]
    assert "grouped_leaf_ff_mma_warp" in names, names
    layer.close()
