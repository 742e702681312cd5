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
