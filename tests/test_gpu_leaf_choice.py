"""Which kernels run: trees of few leaves, where a leaf has hundreds of tiles; thin leaves, whose kernel can walk the whole tree; and
the parity of what is chosen."""
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


@pytest.mark.parametrize("D,depth,B,launches", [
    (256, 12, 7000, 1), (256, 12, 7001, 3), (640, 13, 7000, 1), (640, 13, 7001, 3), (328, 12, 5000, 1), (328, 12, 5001, 3),
    (896, 12, 4608, 1), (896, 12, 4609, 3), (896, 13, 3072, 1), (896, 13, 3073, 2), (896, 13, 4096, 1), (896, 13, 4609, 3),
    (256, 10, 4095, 1), (256, 10, 4096, 5),              # (four tokens per leaf: two stages, a bucketing behind each, the leaves)
])
def test_thin_leaves_walk_the_tree_themselves(D, depth, B, launches):
    cfg = C("thin", D, 64, depth, 1, "relu", "bf16", B, "normal", node_bias_std=0.1)
    case = util.make_case(cfg, seed=2)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    y, leaf = layer.forward_infer(util.to_device(case.x, "bf16"))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    util.check_outputs(y, y_ref, "bf16")
    assert layer.last_launch_count() == launches
    layer.close()


# the three forms of the warp leaf kernel at their lines (148 SMs: 3552 tokens behind a bucketing, 4736 with a walk), rows in vectors
# and not, outputs that fill vectors and not
@pytest.mark.parametrize("D,O,depth,l,B", [
    (64, 48, 12, 1, 4736), (64, 48, 12, 1, 4737), (64, 46, 12, 2, 4737), (64, 48, 12, 4, 900), (64, 48, 12, 3, 4736), (64, 48, 12, 3, 4737),
    (64, 48, 12, 16, 4737), (64, 48, 12, 17, 4737), (63, 48, 12, 3, 4737), (64, 48, 9, 1, 3553), (64, 48, 9, 4, 3553), (64, 48, 9, 8, 3552),
    (64, 48, 9, 8, 3553), (64, 48, 9, 9, 3553), (63, 45, 9, 5, 3553),
])
def test_forms_of_the_warp_leaf_kernel(D, O, depth, l, B):
    cfg = C("forms", D, O, depth, l, "silu", "f32", B, "normal", node_bias_std=0.1)
    case = util.make_case(cfg, seed=6)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    layer.set_path("warp")
    y, leaf = layer.forward_infer(util.to_device(case.x, "f32"))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    util.check_outputs(y, y_ref, "f32")
    layer.close()


def test_the_descent_alone_keeps_its_stages():
    """The walk is the leaf kernel's: fff_tree_descent, behind which there is none, runs the stages."""
    cfg = C("descent_alone", 256, 64, 12, 1, "relu", "bf16", 3000, "normal", node_bias_std=0.1)
    case = util.make_case(cfg, seed=2)
    _, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "bf16")
    np.testing.assert_array_equal(layer.tree_descent(x).cpu().numpy(), leaf_ref)
    assert layer.last_launch_count() == 2                  # two stages, lists between them
    layer.forward_infer(x)
    assert layer.last_launch_count() == 1
    layer.close()
