"""A CTA per token sends for the node rows of its first step before its tokens: widths at both sides of what it keeps in registers
(1024 columns) and trees of fewer levels than a step has."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("D,depth", [(8, 1), (1016, 2), (1024, 3), (1032, 4), (1023, 3)])
def test_the_first_step_matches_the_oracle(D, depth, dtype):
    cfg = wl.FFFConfig("first_step", D, 24, depth, 5, "gelu", dtype, 37, "normal", node_bias_std=0.3)
    case = util.make_case(cfg, seed=6)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, dtype)
    layer.profile_begin(1)
    y, leaf = layer.forward_infer(x)
    torch.cuda.synchronize()
    assert [n for n, _ in layer.profile_end()[0]] == ["forward_token_blocks"]
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    util.check_outputs(y, y_ref, dtype)
    for _ in range(3):                                     # launches one behind the other
        y2, leaf2 = layer.forward_infer(x)
    assert torch.equal(y2, y) and torch.equal(leaf2, leaf)
    layer.close()
