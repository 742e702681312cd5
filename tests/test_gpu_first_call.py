"""The first call of a size on a stream that does not wait for the default stream (every stream that torch makes): what the call
allocates and clears has to be clear before the call's own kernels run.  And what such a call replaces is not read again."""
import pytest
import torch

from paper_2308_14711_b200 import binding, workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
TRAIN = [
    C("first_train_padding", 64, 32, 3, 3, "gelu", "bf16", 400, "normal"),           # 24 hidden columns and 8 weights: 32 columns of padding
    C("first_train_deep", 64, 32, 9, 3, "gelu", "bf16", 400, "normal"),              # node choices and products in separate kernels
]
INFER = [
    C("first_f32_lists", 64, 48, 6, 8, "relu", "f32", 5000, "normal"),               # the leaves' lists and their counts
    C("first_bf16_lists", 128, 64, 7, 16, "gelu", "bf16", 3000, "normal"),
    C("first_bf16_node_lists", 128, 64, 10, 16, "gelu", "bf16", 6000, "normal"),     # two stages with lists between them
    C("first_bf16_block_sums", 128, 64, 4, 72, "gelu", "bf16", 9000, "normal"),
]


def on_a_side_stream(call):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        out = call()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("cfg", TRAIN, ids=lambda c: c.name)
def test_first_forward_train_on_a_side_stream(cfg):
    case = util.make_case(cfg, seed=2, margin=None)
    x = util.to_device(case.x, cfg.dtype)
    for _ in range(4):
        layer = util.make_layer(case)
        first = on_a_side_stream(lambda: layer.forward_train(x))
        again = layer.forward_train(x)
        torch.cuda.synchronize()
        assert layer.last_status() == 0
        for a, b in zip(first, again):
            assert torch.equal(a, b)
        layer.close()


@pytest.mark.parametrize("cfg", INFER, ids=lambda c: c.name)
def test_first_forward_infer_on_a_side_stream(cfg):
    case = util.make_case(cfg, seed=2)
    x = util.to_device(case.x, cfg.dtype)
    for _ in range(4):
        layer = util.make_layer(case)
        small = on_a_side_stream(lambda: layer.forward_infer(x[: cfg.B // 3]))       # then the larger batch grows the workspace
        first = on_a_side_stream(lambda: layer.forward_infer(x))
        again = layer.forward_infer(x)
        torch.cuda.synchronize()
        assert layer.last_status() == 0
        for a, b, c in zip(first, again, small):
            assert torch.equal(a, b)
            assert a.dtype != torch.int32 or torch.equal(a[: cfg.B // 3], c)
        layer.close()


@pytest.mark.parametrize("B", [100, 4000])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_no_bucketing_once_its_buffers_are_gone(dtype, B):
    """The bucketing of the last forward is made on demand from buffers that a larger batch replaces."""
    cfg = C("gone", 128, 64, 5, 8, "relu", dtype, B, "normal")
    case = util.make_case(cfg, seed=1)
    layer = util.make_layer(case)
    x = util.to_device(case.x, dtype)
    layer.forward_infer(x)
    layer.reserve(20000)
    with pytest.raises(binding.FFFError) as e:
        layer.last_bucketing(B)
    assert e.value.status == 1
    _, leaf = layer.forward_infer(x)
    _, perm = layer.last_bucketing(B)
    assert torch.equal(perm.long(), torch.argsort(leaf.long(), stable=True))
    layer.close()


def test_no_bucketing_from_staging_buffers_that_are_gone():
    """A host-buffer forward in chunks, then one whose staging buffers cannot be allocated."""
    cfg = C("gone_staging", 1024, 1024, 3, 8, "relu", "bf16", 1200, "normal")
    case = util.make_case(cfg, seed=1)
    layer = util.make_layer(case)
    xh = util.to_device(case.x, "bf16").cpu().pin_memory()
    yh, lh = torch.empty_like(xh), torch.empty(cfg.B, dtype=torch.int32)
    layer.forward_infer_host(xh, yh, lh)
    too_many = 1 << 27                                     # 256 GiB of rows: the host pointers are not looked at
    status = binding.lib().fff_forward_infer_host(layer._h, xh.data_ptr(), yh.data_ptr(), lh.data_ptr(), too_many, None)
    assert binding.STATUS_NAMES[status] in ("FFF_ERR_ALLOC", "FFF_ERR_UNSUPPORTED")
    with pytest.raises(binding.FFFError) as e:
        layer.last_bucketing(cfg.B)
    assert e.value.status == 1
    layer.forward_infer_host(xh, yh, lh)
    _, perm = layer.last_bucketing(cfg.B)
    assert torch.equal(perm.cpu().long(), torch.argsort(lh.long(), stable=True))
    layer.close()
