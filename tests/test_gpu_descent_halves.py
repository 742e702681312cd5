"""First descent stage with two CTAs per tile, one for each half of the tree below the root: routing against the oracle at the
sizes where the form starts, ends and leaves ragged tiles."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [7, 8, 14])
@pytest.mark.parametrize("D,B", [(128, 1), (128, 513), (200, 3152), (128, 9472), (128, 9473)])
def test_halves_route_as_the_oracle(depth, D, B):
    """9472 = 74 tiles of 128: the last size with two CTAs per tile on 148 SMs.  depth 14: the 8-level first stage of three."""
    cfg = wl.FFFConfig("halves", D, 64, depth, 8, "gelu", "bf16", B, "normal", node_bias_std=0.3)
    case = util.make_case(cfg, seed=6)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    layer.set_tuning("token_blocks", False)
    x = util.to_device(case.x, cfg.dtype)
    for _ in range(2):                                     # the second call starts from the counts the first one cleared
        y, leaf = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_status() == 0
        np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
        util.check_outputs(y, y_ref, cfg.dtype)
    layer.close()


@pytest.mark.parametrize("depth", [7, 8])
def test_ties_and_nan_at_the_root(depth):
    """Zero node weights: every logit is 0 and every token goes right; NaN rows go left at every node, in one half only."""
    D, l, B, n = 128, 8, 600, 1 << depth
    z = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device="cuda")
    from paper_2308_14711_b200 import binding
    layer = binding.FFFLayer(D, 64, depth, l, "relu", "bf16", z(n - 1, D), z(n - 1), z(n, l, D), z(n, l), z(n, 64, l), z(n, 64))
    layer.set_tuning("token_blocks", False)
    x = torch.ones(B, D, dtype=torch.bfloat16, device="cuda")
    x[::3] = float("nan")
    _, leaf = layer.forward_infer(x)
    want = torch.full((B,), n - 1, dtype=torch.int32)
    want[::3] = 0
    assert torch.equal(leaf.cpu(), want)
    layer.close()
