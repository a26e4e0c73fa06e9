"""The search call's native side: a file of its own for every Python and torch, without which the library works all the same."""
import os
import sysconfig

import pytest
import torch

from paper_2502_08923_b200 import binding as cs, build


@pytest.fixture
def fresh(monkeypatch):
    """The binding as it is before the library is loaded (which is built and up to date)."""
    cs.load()
    monkeypatch.setattr(cs, "_lib", None)
    monkeypatch.setattr(cs, "_search", None)
    return monkeypatch


def test_is_built_for_this_python_and_torch(fresh):
    name = os.path.basename(build.native_path())
    assert sysconfig.get_config_var("SOABI") in name and torch.__version__ in name
    cs.load(build_if_missing=False)
    assert type(cs._search) is type(len)


@pytest.mark.parametrize("content", [None, b"not a module"])
def test_the_general_path_stands_in(content, fresh, tmp_path):
    path = tmp_path / "_native.so"
    if content is not None:
        path.write_bytes(content)
    fresh.setattr(build, "native_path", lambda: str(path))
    with pytest.warns(RuntimeWarning, match="general path"):
        lib = cs.load(build_if_missing=False)
    assert lib.cs_find_match(None, None, 0, 0, 3, 10, 0, None, None, None, None) == cs.CS_OK
    with pytest.raises(ValueError, match="contiguous CUDA tensor"):
        cs.cs_find_match(torch.zeros(1, 16, dtype=torch.int32), torch.zeros(1, dtype=torch.int32), 3, 4)


@pytest.mark.parametrize("compiler", ["false", "/nonexistent/g++"])
def test_a_host_that_cannot_build_it(compiler, fresh, tmp_path):
    """The library itself is up to date and is left alone; an older file of the native side does not stay."""
    path = tmp_path / "_native.so"
    path.write_bytes(b"older than its source")
    os.utime(path, (0, 0))
    fresh.setattr(build, "native_path", lambda: str(path))
    fresh.setenv("CXX", compiler)
    fresh.setenv("NVCC", "/nonexistent/nvcc")
    with pytest.warns(RuntimeWarning, match="general path"):
        assert build.build() == build.LIB
    assert os.listdir(tmp_path) == []
