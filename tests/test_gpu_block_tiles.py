"""The one-launch kernel on bulk copies (float32 layers), where it is chosen: sizes at which its tiles, blocks of weights and copies have
remainders.

Rows that start between 16-byte boundaries (input and output widths that are no multiple of 4), one to four tokens per warp in the
descent and more than one round of it, tiles of 8, 16 and 32 tokens, leaves whose weights take one block and several, fewer than
eight units in the last block, one to four outputs per thread, a ring of two slots; next to sizes that are left to the other one-launch kernel or
do not fit this one.  The same bits as a warp per token (the sums are added in the same order)."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
TILES = [
    C("bt_d3_narrow", 784, 10, 3, 32, "relu", "f32", 600, "normal"),
    C("bt_one_leaf", 129, 30, 0, 40, "gelu", "f32", 700, "normal"),
    C("bt_d1", 133, 2, 1, 60, "gelu", "f32", 2600, "normal", node_bias_std=0.3),
    C("bt_d1_rounds", 255, 3, 1, 64, "gelu", "f32", 10007, "normal", node_bias_std=0.3),
    C("bt_d2_ragged", 130, 5, 2, 40, "silu", "f32", 12000, "normal"),
    C("bt_d6_short_rows", 107, 20, 6, 52, "gelu", "f32", 1210, "normal"),
    C("bt_d6_two_outputs", 387, 259, 6, 33, "gelu", "f32", 4700, "normal"),
    C("bt_d8_three_tokens", 768, 768, 8, 12, "gelu", "f32", 6304, "layernorm"),
    C("bt_d8_three_outputs", 768, 768, 8, 12, "gelu", "f32", 3000, "layernorm"),
    C("bt_d4_wide", 1024, 1024, 4, 33, "gelu_tanh", "f32", 1500, "normal"),
    C("bt_d4_ragged_wide", 1021, 1023, 4, 20, "gelu", "f32", 1300, "normal"),
    C("bt_d3_rounds", 1001, 901, 3, 12, "gelu", "f32", 12000, "clusters"),
    C("bt_d9_rounds", 768, 768, 9, 16, "gelu", "f32", 10007, "clusters"),
    C("bt_d3_long_rows", 1300, 40, 3, 8, "gelu", "f32", 900, "normal"),
    C("bt_d3_two_slots", 2056, 40, 3, 8, "gelu", "f32", 900, "normal"),
]
OTHERS = [
    C("bt_d3_too_long", 2600, 40, 3, 8, "gelu", "f32", 900, "normal"),
    C("bt_d2_too_many_outputs", 64, 1100, 2, 8, "gelu", "f32", 900, "normal"),
    C("bt_d2_many_outputs", 130, 1024, 4, 12, "gelu", "f32", 1200, "normal"),
    C("bt_tiny", 5, 3, 0, 1, "gelu", "f32", 700, "normal"),
    C("bt_d1_tiny", 33, 1, 1, 4, "gelu", "f32", 2501, "normal", node_bias_std=0.3),
    C("bt_d6_many_outputs", 130, 257, 6, 9, "gelu", "f32", 6304, "normal"),
    C("bt_d5_many", 64, 48, 5, 16, "relu", "f32", 20011, "clusters"),
    C("bt_d9_empty_leaves", 72, 520, 9, 12, "gelu", "f32", 6000, "clusters"),
    C("bt_d9_thin", 256, 256, 9, 8, "gelu", "f32", 1500, "normal"),
]


def kernels_of(layer, x):
    """Names of the kernels that a forward launches, from a recording of it (both kernels run under one name in the library's own list)."""
    from cuda.bindings import driver

    def call(f, *args):
        error, *result = f(*args)
        assert error == driver.CUresult.CUDA_SUCCESS, (f, error)
        return result
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        layer.forward_infer(x)
    raw = driver.CUgraph(init_value=graph.raw_cuda_graph())
    nodes, count = call(driver.cuGraphGetNodes, raw, 64)
    names = []
    for node in nodes[:count]:
        if call(driver.cuGraphNodeGetType, node)[0] == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            params = call(driver.cuGraphKernelNodeGetParams, node)[0]
            by_kernel = int(params.func) == 0
            names += call(driver.cuKernelGetName, params.kern) if by_kernel else call(driver.cuFuncGetName, params.func)
    return [n.decode() for n in names]


@pytest.mark.parametrize("cfg,kernel", [(c, "k_block_tiles") for c in TILES] + [(c, "k_block_forward") for c in OTHERS],
                         ids=lambda v: getattr(v, "name", ""))
def test_block_tiles_match_the_oracle(cfg, kernel):
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
    names = kernels_of(layer, x)
    assert len(names) == 1 and kernel in names[0]
    layer.set_path("warp")
    y2, leaf2 = layer.forward_infer(x)
    assert torch.equal(y2, y) and torch.equal(leaf2, leaf)
    layer.close()
