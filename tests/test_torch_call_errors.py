"""The tensor-level call when asking a tensor about itself fails: a Python error, as from any other call (no GPU work)."""
import pytest
import torch

from paper_2308_14711_b200 import binding, build


@pytest.fixture(scope="module")
def forward():
    build.build()
    return binding.torch_call().forward


class Unreadable(torch.Tensor):
    """Says that it lives on the GPU; every operator on it, strides and contiguity among them, raises."""

    @staticmethod
    def __new__(cls, rows, cols):
        return torch.Tensor._make_wrapper_subclass(cls, (rows, cols), dtype=torch.float32, device="cuda",
                                                   dispatch_sizes_strides_policy="strides")

    @classmethod
    def __torch_dispatch__(cls, func, types, args=(), kwargs=None):
        raise KeyError(f"no {func}")


def test_an_error_of_a_tensor_is_raised_to_the_caller(forward):
    bad = Unreadable(4, 8)
    with pytest.raises(KeyError, match="no aten"):
        forward(0, 8, 4, False, bad, None, None, True, 0)


def test_arguments_that_are_not_taken_give_none(forward):
    x = torch.zeros(4, 8)
    assert forward(0, 8, 4, False, x, None, None, True, 0) is None                     # not on the GPU
    assert forward(0, 8, 4, False, x.to_sparse_csr(), None, None, True, 0) is None
    assert forward(0, 8, 4, False, "x", None, None, True, 0) is None
    assert forward(0, 8, 4, False, torch.zeros(()), None, None, True, 0) is None
