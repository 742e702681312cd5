"""GPU parity of bf16 layers whose input width is a multiple of 8 but not of 128: the tensor-core kernels run on weight
images padded with zero columns, and the padding columns of the token rows are zeros made by the copy engine (tcgen05
kernels) or by the copy instructions (mma.sync kernels).  Against the oracle, at the edges of the padding (8 and 120
columns short of a multiple of 128, exactly 64) and through every kernel that takes padded rows."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
CASES = [
    C("pad_136_one_stage", 136, 128, 5, 16, "gelu", "bf16", 3000, "normal"),          # tcgen05 descent and leaves, no bucketing
    C("pad_248_pairs", 248, 64, 7, 12, "relu", "bf16", 20001, "normal"),              # first stage on CTA pairs
    C("pad_192_thin", 192, 72, 7, 24, "silu", "bf16", 700, "normal"),                 # thin buckets: mma.sync leaves; a whole K-block of padding
    C("pad_1016_two_stages", 1016, 48, 10, 16, "gelu", "bf16", 20000, "clusters"),    # grouped second stage, node lists
    C("pad_200_two_stages_mma", 200, 40, 9, 20, "gelu", "bf16", 1500, "normal"),      # second stage on mma.sync
    C("pad_264_group_tiles", 264, 80, 9, 12, "gelu", "bf16", 9000, "normal"),         # tiles of eight sibling leaves
    C("pad_328_deep", 328, 32, 11, 1, "gelu", "bf16", 4000, "normal"),                # warp leaves behind tensor-core stages
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_padded_width_matches_the_oracle(cfg):
    case = util.make_case(cfg, seed=4)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    assert layer.capabilities() & 128 and not layer.capabilities() & (1 | 2 | 4 | 8)
    # rows of x are followed by non-finite values in memory: the padding must not read into the next row or past the end
    guard = torch.full((cfg.B + 1, cfg.D), float("nan"), dtype=torch.bfloat16, device="cuda")
    guard[:cfg.B] = util.to_device(case.x, "bf16")
    x = guard[:cfg.B]
    for tuned in (True, False):
        for key in ("tcgen05_descent", "tcgen05_leaf"):
            layer.set_tuning(key, tuned)
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_status() == 0
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        util.check_outputs(y, y_ref, "bf16")
    layer.close()


PRECISE = CASES + [
    C("pad_328_warp_tiles", 328, 272, 9, 13, "silu", "bf16", 5001, "normal"),         # a warp per tile
    C("pad_200_l64", 200, 64, 4, 64, "gelu", "bf16", 9000, "normal"),                 # widest leaves, no spare column for the bias
    C("pad_200_l40", 200, 64, 4, 40, "relu", "bf16", 9000, "clusters"),
    C("pad_200_l33_mma", 200, 64, 4, 33, "gelu_tanh", "bf16", 1000, "normal"),
    C("pad_136_l32", 136, 144, 3, 32, "relu", "bf16", 12000, "normal"),
    C("pad_136_l32_mma", 136, 144, 5, 32, "gelu", "bf16", 2000, "normal"),
]


@pytest.mark.parametrize("cfg", PRECISE, ids=lambda c: c.name)
def test_padded_layers_keep_the_hidden_values_precision(cfg):
    """Rounding the output to bf16 is the only rounding that shows: next to no value differs from the oracle's, rounded.

    A hidden value is within 2^-18 of its float32 value, so y is off by about 2^-19 of the root of its summed squares before it is
    rounded to steps of 2^-8 to 2^-7 of itself: about one value in 1000 of that size falls on the other side of a step, more of the
    small ones.  With hidden values rounded to bf16 (2^-9) it is four in ten."""
    case = util.make_case(cfg, seed=5)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "bf16")
    want = torch.from_numpy(y_ref).to(torch.bfloat16)
    for off in ((), ("token_blocks",), ("token_blocks", "tcgen05_leaf"), ("token_blocks", "direct_lists")):
        for key in off:
            layer.set_tuning(key, False)
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        for key in off:
            layer.set_tuning(key, True)
        assert float((y.cpu() != want).float().mean()) < 0.03
    layer.close()


@pytest.mark.parametrize("depth,l,B", [(5, 16, 3000), (4, 12, 20000), (9, 12, 9000), (9, 13, 5001), (3, 40, 3000)])
def test_infinite_hidden_values_reach_the_output(depth, l, B):
    """A hidden value past the largest bf16 is infinite, not NaN: y is +inf where its weight is positive."""
    D, O, n = 136, 48, 1 << depth
    full = lambda v, *s: torch.full(s, v, dtype=torch.bfloat16, device="cuda")
    from paper_2308_14711_b200 import binding
    layer = binding.FFFLayer(D, O, depth, l, "relu", "bf16", full(1.0, n - 1, D), full(0.0, n - 1), full(3e38, n, l, D), full(0.0, n, l),
                             full(1.0, n, O, l), full(0.0, n, O))
    y, _ = layer.forward_infer(full(1.0, B, D))
    assert bool(torch.isposinf(y).all())
    layer.close()
