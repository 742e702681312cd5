"""What the build looks for and what it names its files (no compiler runs, no GPU work)."""
import os

import torch

from paper_2308_14711_b200 import build


def test_the_module_of_another_torch_is_another_file(monkeypatch):
    here = build.call_lib()
    assert os.path.dirname(here) == os.path.dirname(build.LIB) and here.endswith(".so") and torch.__version__ in here
    monkeypatch.setattr(torch, "__version__", "9.9.9+cu999")
    assert build.call_lib() != here and "9.9.9+cu999" in build.call_lib()


def test_the_toolkit_of_a_bare_compiler_name(monkeypatch, tmp_path):
    nvcc = tmp_path / "toolkit" / "bin" / "nvcc"
    nvcc.parent.mkdir(parents=True)
    nvcc.write_text("#!/bin/sh\n")
    nvcc.chmod(0o755)
    for name in (str(nvcc), "nvcc"):
        monkeypatch.setattr(build, "NVCC", name)
        monkeypatch.setenv("PATH", str(nvcc.parent))
        assert build.cuda_home() == os.path.realpath(tmp_path / "toolkit")


def test_the_library_is_built_where_the_module_cannot_be(monkeypatch):
    def no_compiler(force=False):
        raise OSError("no g++")
    monkeypatch.setattr(build, "build_call", no_compiler)
    monkeypatch.setattr(build, "up_to_date", lambda: True)
    import pytest
    with pytest.warns(UserWarning, match="through ctypes"):
        assert build.build() == build.LIB
