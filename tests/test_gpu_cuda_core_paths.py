"""GPU parity of the two one-launch kernels on CUDA cores against the oracle, at the sizes where they can go wrong.

Token blocks (a CTA per token): depths around the three levels of a step, rows that are no multiple of 16 bytes, output
weights staged in several parts or not 16-byte aligned, leaves wider than the sixteen units of a pass.
Block forward (descent, grid barrier, tiles of 8 or 16 tokens of a leaf): one and four tokens per warp in the descent, tiles
with a remainder, narrow outputs that share a tile's tokens out, all tokens in one leaf."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
TOKEN_BLOCKS = [
    C("tb_d0", 40, 24, 0, 5, "gelu", "f32", 3, "normal"),
    C("tb_d1_scalar_rows", 37, 3, 1, 1, "relu", "f32", 200, "normal", node_bias_std=0.5),
    C("tb_d3", 784, 10, 3, 32, "relu", "f32", 130, "normal"),
    C("tb_d4_long_rows", 2056, 40, 4, 17, "silu", "f32", 150, "normal"),             # more than 1024 columns
    C("tb_d8_staged_twice", 256, 1030, 8, 40, "gelu", "bf16", 300, "normal"),        # 82 KB of output weights per leaf
    C("tb_d7_unaligned_w2", 72, 7, 7, 3, "gelu_tanh", "bf16", 64, "normal"),         # 42-byte output matrices
    C("tb_d15", 128, 64, 15, 1, "gelu", "bf16", 257, "normal"),
    C("tb_d10_two_stages", 128, 64, 10, 16, "gelu", "bf16", 1184, "clusters"),           # the most tokens it is taken for on 148 SMs
    C("tb_ragged_bf16", 101, 36, 5, 7, "gelu", "bf16", 100, "normal", node_bias_std=0.2),
]
BLOCKS = [
    C("bf_d3_narrow", 784, 10, 3, 32, "relu", "f32", 2048, "normal"),                # tiles of 8, two tokens per thread in the output layer
    C("bf_d0", 64, 300, 0, 9, "gelu", "f32", 700, "normal"),
    C("bf_d1", 33, 1, 1, 1, "gelu", "f32", 650, "normal", node_bias_std=0.5),
    C("bf_d5_four_tokens", 200, 70, 5, 10, "silu", "f32", 5003, "normal"),
    C("bf_d9_skew", 96, 520, 9, 12, "gelu", "f32", 6000, "clusters"),                # tiles of 16, empty leaves
    C("bf_d2_wide_leaf", 61, 130, 2, 70, "gelu_tanh", "f32", 5000, "normal"),
    C("bf_bf16_odd", 100, 36, 3, 33, "gelu", "bf16", 5000, "normal", node_bias_std=0.2),
    C("bf_bf16_wide_leaf", 128, 64, 4, 80, "relu", "bf16", 900, "normal"),           # l > 64: no tensor-core leaf kernel
]


def check(cfg, switch, seed):
    case = util.make_case(cfg, seed=seed)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    off_ref, perm_ref = orc.bucket(leaf_ref, cfg.n_leaves)
    layer = util.make_layer(case)
    x = util.to_device(case.x, cfg.dtype)
    y_first = None
    for _ in range(2):                                     # the second call starts from the counts the first one cleared
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_launch_count() == 1 and layer.last_status() == 0
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        util.check_outputs(y, y_ref, cfg.dtype)
        assert y_first is None or torch.equal(y, y_first)
        y_first = y
    off, perm = layer.last_bucketing(cfg.B)
    np.testing.assert_array_equal(off.cpu().numpy(), off_ref)
    np.testing.assert_array_equal(perm.cpu().numpy(), perm_ref)
    layer.set_tuning(switch, False)
    y2, leaf2 = layer.forward_infer(x)
    np.testing.assert_array_equal(leaf2.cpu().numpy(), leaf_ref)
    util.check_outputs(y2, y_ref, cfg.dtype)
    layer.close()


@pytest.mark.parametrize("cfg", TOKEN_BLOCKS, ids=lambda c: c.name)
def test_token_blocks_match_the_oracle(cfg):
    check(cfg, "token_blocks", seed=7)


@pytest.mark.parametrize("cfg", BLOCKS, ids=lambda c: c.name)
def test_block_forward_matches_the_oracle(cfg):
    check(cfg, "fused_small", seed=8)


def launches_of(layer, x):
    layer.profile_begin(1)
    layer.forward_infer(x)
    torch.cuda.synchronize()
    return [n for n, _ in layer.profile_end()[0]]


def test_the_batches_served_before_do_not_choose_the_kernel():
    """4096 leaves: the lists of more than 65 536 tokens would pass 1 GiB."""
    cfg = C("bf_state", 32, 24, 12, 32, "gelu", "f32", 2000, "normal")
    case = util.make_case(cfg, seed=3)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "f32")
    names = launches_of(layer, x)
    y, leaf = layer.forward_infer(x)
    layer.reserve(70000)
    assert launches_of(layer, x) == names == ["fused_forward_blocks"]
    y2, leaf2 = layer.forward_infer(x)
    assert torch.equal(y, y2) and torch.equal(leaf, leaf2)
    layer.close()


@pytest.mark.parametrize("pin_first", [True, False])
def test_batches_past_the_lists_run_in_parts(pin_first):
    cfg = C("bf_parts", 16, 24, 12, 1, "relu", "f32", 65536 + 1603, "normal", node_bias_std=0.1)
    case = util.make_case(cfg, seed=4)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    off_ref, perm_ref = orc.bucket(leaf_ref, cfg.n_leaves)
    layer = util.make_layer(case, path="fused" if pin_first else "auto")
    x = util.to_device(case.x, "f32")
    if not pin_first:
        layer.set_path("warp")
        layer.reserve(cfg.B)
        layer.set_path("fused")
    for _ in range(2):
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_launch_count() == 2
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        util.check_outputs(y, y_ref, "f32")
    off, perm = layer.last_bucketing(cfg.B)
    np.testing.assert_array_equal(off.cpu().numpy(), off_ref)
    np.testing.assert_array_equal(perm.cpu().numpy(), perm_ref)
    layer.set_path("warp")                                 # one warp per token: the same sums in the same order
    y2, leaf2 = layer.forward_infer(x)
    assert torch.equal(y2, y) and torch.equal(leaf2, leaf)
    layer.close()


def test_two_handles_on_two_streams():
    """Grids of all SMs with a barrier each, enqueued on two streams at the same time."""
    cfgs = [C("bf_stream_a", 200, 70, 5, 10, "silu", "f32", 5003, "normal"), C("bf_stream_b", 784, 10, 3, 32, "relu", "f32", 4100, "normal")]
    streams = [torch.cuda.Stream() for _ in cfgs]
    layers, xs, refs = [], [], []
    for i, cfg in enumerate(cfgs):
        case = util.make_case(cfg, seed=5 + i)
        layers.append(util.make_layer(case))
        xs.append(util.to_device(case.x, "f32"))
        refs.append(layers[i].forward_infer(xs[i]))
    torch.cuda.synchronize()
    outs = [[], []]
    for _ in range(20):
        for i, layer in enumerate(layers):
            with torch.cuda.stream(streams[i]):
                outs[i].append(layer.forward_infer(xs[i]))
    torch.cuda.synchronize()
    for layer, got, (y, leaf) in zip(layers, outs, refs):
        assert layer.last_status() == 0
        for y2, leaf2 in got:
            assert torch.equal(y2, y) and torch.equal(leaf2, leaf)
        layer.close()


# tokens per leaf and neurons at both sides of the line; either kernel adds a token's sums in the same order
@pytest.mark.parametrize("depth,l,B,kernel", [
    (9, 8, 1024, "fused_forward_blocks"), (9, 8, 1023, "descent_tail+leaf_ff_warp"), (10, 16, 1024, "fused_forward_blocks"),
    (10, 16, 1023, "descent_tail+leaf_ff_warp"), (10, 7, 4096, "grouped_leaf_ff_warp"), (10, 8, 4096, "fused_forward_blocks"),
    (10, 3, 10240, "fused_forward_blocks"), (10, 3, 10239, "grouped_leaf_ff_warp"), (11, 3, 20480, "grouped_leaf_ff_warp"),
    (11, 4, 20480, "fused_forward_blocks"), (8, 1, 1024, "fused_forward_blocks"), (8, 1, 1023, "descent_tail+leaf_ff_warp"),
])
def test_thin_leaves_with_few_tokens_keep_a_warp_per_token(depth, l, B, kernel):
    cfg = C("bf_line", 40, 24, depth, l, "gelu", "f32", B, "normal", node_bias_std=0.1)
    case = util.make_case(cfg, seed=3)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "f32")
    assert launches_of(layer, x)[-1] == kernel
    y, leaf = layer.forward_infer(x)
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    util.check_outputs(y, y_ref, "f32")
    layer.set_tuning("fused_small", kernel != "fused_forward_blocks")
    if kernel == "fused_forward_blocks":
        y2, leaf2 = layer.forward_infer(x)
        assert launches_of(layer, x)[-1] != kernel and torch.equal(y2, y) and torch.equal(leaf2, leaf)
    layer.close()


@pytest.mark.parametrize("D,O,depth,l,B", [(768, 64, 5, 12, 300), (101, 37, 7, 7, 500), (64, 48, 8, 33, 200), (72, 40, 3, 1, 450)])
def test_float32_gives_the_same_bits_on_every_kernel(D, O, depth, l, B):
    cfg = C("same_bits", D, O, depth, l, "gelu", "f32", B, "normal", node_bias_std=0.2)
    case = util.make_case(cfg, seed=8)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "f32")
    y, leaf = layer.forward_infer(x)                       # a CTA per token
    half, _ = layer.forward_infer(x[: B // 2].contiguous())
    assert layer.last_launch_count() == 1 and torch.equal(half, y[: B // 2])
    for key in ("token_blocks", "fused_small"):            # the one-launch kernel, a warp per token
        layer.set_tuning(key, False)
        y2, leaf2 = layer.forward_infer(x)
        assert torch.equal(y2, y) and torch.equal(leaf2, leaf)
    big, _ = layer.forward_infer(x.repeat(13, 1))
    assert torch.equal(big[:B], y) and torch.equal(big[-B:], y)
    layer.close()
