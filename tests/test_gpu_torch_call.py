"""Tensor-level forward_infer: what it allocates, what it returns, and the errors of arguments it does not take."""
import pytest
import torch

from paper_2308_14711_b200 import binding

pytestmark = pytest.mark.gpu

D, O, DEPTH, LW = 64, 24, 3, 4


def make(dtype):
    g = torch.Generator().manual_seed(3)
    rnd = lambda *s: (torch.randn(*s, generator=g) * 0.2).to(dtype).cuda()
    return binding.FFFLayer(D, O, DEPTH, LW, "gelu", "bf16" if dtype == torch.bfloat16 else "f32", rnd(7, D), rnd(7), rnd(8, LW, D), rnd(8, LW), rnd(8, O, LW), rnd(8, O))


@pytest.fixture(params=["module", "ctypes"])
def call(request, monkeypatch):
    """The call through the CPython module, and as it is made where that has not been built."""
    if request.param == "ctypes":
        monkeypatch.setattr(binding, "torch_call", lambda: None)
    else:
        assert binding.torch_call() is not None


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("B", [0, 1, 5])
def test_buffers_and_results(call, dtype, B):
    layer = make(dtype)
    x = torch.randn(B, D, device="cuda").to(dtype).requires_grad_(dtype == torch.float32)
    y, leaf = layer.forward_infer(x)
    assert y.shape == (B, O) and y.dtype == dtype and not y.requires_grad
    assert leaf.shape == (B,) and leaf.dtype == torch.int32
    y2, none = layer.forward_infer(x, want_leaf_idx=False)
    assert none is None
    ybuf, lbuf = torch.full_like(y, 7), torch.full_like(leaf, -1)
    got = layer.forward_infer(x, ybuf, lbuf)
    assert got[0] is ybuf and got[1] is lbuf
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        y3, leaf3 = layer.forward_infer(x)
    y4, _ = layer.forward_infer(x, stream=side)
    torch.cuda.synchronize()
    for other in (y2, ybuf, y3, y4):
        assert torch.equal(other, y)
    assert torch.equal(lbuf, leaf) and torch.equal(leaf3, leaf)


def test_wrong_arguments_name_themselves(call):
    layer = make(torch.float32)
    x = torch.randn(4, D, device="cuda")
    y = torch.empty(4, O, device="cuda")
    for bad in (x.cpu(), x.bfloat16(), x[:, :-1], x.t().contiguous().t(), torch.randn(4, D + 1, device="cuda")):
        with pytest.raises(ValueError, match="^x: expected"):
            layer.forward_infer(bad)
    for bad in (x.to_sparse_csr(), x.to_sparse()):         # these raise when asked whether they are contiguous, or are not
        with pytest.raises((RuntimeError, ValueError)):
            layer.forward_infer(bad)
    with pytest.raises(ValueError, match="^y: expected"):
        layer.forward_infer(x, y[:3])
    with pytest.raises(ValueError, match="^leaf_idx: expected"):
        layer.forward_infer(x, y, torch.zeros(4, dtype=torch.int64, device="cuda"))
    layer.close()
    with pytest.raises(binding.FFFError):
        layer.forward_infer(x)
