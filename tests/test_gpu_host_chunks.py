"""Host-buffer forwards of small batches, cut into chunks by the bytes they copy: the same bits as an unchunked forward."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu


# two chunks from 4 MB of x and y on (3907 tokens of 1024 bytes); the later cases: chunks that alone would run as token
# blocks, weights that would be fetched again (one chunk), thin leaves, grouped tiles for the whole batch only, float32
@pytest.mark.parametrize("D,O,depth,l,dtype,B", [
    (256, 256, 4, 12, "bf16", 3906), (256, 256, 4, 12, "bf16", 3907), (1024, 1024, 3, 8, "bf16", 1001),
    (768, 768, 9, 24, "bf16", 1400), (768, 768, 11, 1, "bf16", 3000), (256, 256, 9, 12, "bf16", 8300), (512, 512, 4, 8, "f32", 1500),
    # chunks that alone would run fewer descent stages (12 and 14 tokens per group of the second), thin groups on other kernels,
    # a walk through all levels
    (768, 768, 11, 12, "bf16", 1490), (768, 768, 11, 12, "bf16", 1600), (768, 768, 10, 24, "bf16", 3000), (768, 768, 15, 1, "bf16", 12000),
])
def test_small_batches_in_chunks(D, O, depth, l, dtype, B):
    cfg = wl.FFFConfig("host_small_chunks", D, O, depth, l, "gelu", dtype, B, "normal")
    case = util.make_case(cfg, seed=4)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    xh = torch.from_numpy(case.x).to(td).pin_memory()
    yh = torch.zeros((B, O), dtype=td).pin_memory()
    lh = torch.full((B,), -1, dtype=torch.int32).pin_memory()
    layer.forward_infer_host(xh, yh, lh)
    launches = layer.last_launch_count()                   # (of the last chunk)
    np.testing.assert_array_equal(lh.numpy(), leaf_ref)
    util.check_outputs(yh, y_ref, dtype)
    offsets, perm = layer.last_bucketing(B)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(perm.cpu().numpy(), np.argsort(leaf_ref, kind="stable"))
    assert int(offsets[-1]) == B
    y_dev, _ = layer.forward_infer(xh.cuda())
    torch.cuda.synchronize()
    assert torch.equal(y_dev.cpu(), yh)
    assert layer.last_launch_count() == launches           # a chunk runs what the whole batch runs
    layer.close()


@pytest.mark.parametrize("pinned_x,pinned_y", [(True, True), (False, False), (True, False), (False, True)])
def test_pageable_and_pinned_buffers_give_the_same(pinned_x, pinned_y):
    cfg = wl.FFFConfig("host_pageable", 768, 768, 6, 12, "gelu", "bf16", 3000, "normal")
    case = util.make_case(cfg, seed=4)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "bf16")
    y_dev, leaf_dev = layer.forward_infer(x)
    xh = x.cpu()
    yh = torch.zeros((cfg.B, cfg.O), dtype=torch.bfloat16)
    lh = torch.full((cfg.B,), -1, dtype=torch.int32)
    if pinned_x:
        xh = xh.pin_memory()
    if pinned_y:
        yh, lh = yh.pin_memory(), lh.pin_memory()
    layer.forward_infer_host(xh, yh, lh)
    assert torch.equal(yh, y_dev.cpu()) and torch.equal(lh, leaf_dev.cpu())
    layer.close()
