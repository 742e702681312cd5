"""Which leaf kernel runs: trees of few leaves, where a leaf has hundreds of tiles, and the parity of what is chosen."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
MMA, UMMA = "grouped_leaf_ff_mma", "grouped_leaf_ff_umma"


# 32- and 64-row tiles of all leaves fit 148 SMs with two CTAs (leaves of up to 32 neurons) up to about 18 000 tokens
@pytest.mark.parametrize("depth,l,B,kernel", [
    (0, 12, 50432, UMMA), (0, 24, 50432, UMMA), (0, 48, 50432, UMMA), (1, 12, 50432, UMMA), (1, 48, 50432, UMMA),
    (2, 12, 50432, UMMA), (2, 24, 50432, UMMA), (2, 24, 20000, UMMA), (2, 12, 3000, MMA), (0, 12, 3000, MMA),
])
def test_trees_of_few_leaves(depth, l, B, kernel):
    cfg = C("few_leaves", 128, 64, depth, l, "gelu", "bf16", B, "normal", node_bias_std=0.1)
    case = util.make_case(cfg, seed=2)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "bf16")
    layer.profile_begin(1)
    y, leaf = layer.forward_infer(x)
    torch.cuda.synchronize()
    names = [n for n, _ in layer.profile_end()[0]]
    assert names[-1] == kernel, names
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    util.check_outputs(y, y_ref, "bf16")
    layer.close()
