"""The C-ABI library builds for sm_103a, loads, and exports every function include/tersoff.h declares
(no compute calls: these tests run without a GPU)."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def header_functions():
    src = open(os.path.join(ROOT, "include", "tersoff.h")).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(tersoff_[a-z_]+)\s*\(", src)))


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11474_gb300 import build
    path = build.build()
    return ctypes.CDLL(path)


def test_header_declares_the_boundary_calls():
    names = header_functions()
    for required in ("tersoff_build_neighbors", "tersoff_eval", "tersoff_fitness", "tersoff_param_grad"):
        assert required in names


def test_library_exports_every_declared_symbol(lib):
    for name in header_functions():
        assert hasattr(lib, name), name


def test_binding_covers_every_declared_symbol():
    from paper_1909_11474_gb300 import binding
    assert sorted(binding.EXPORTED) == header_functions()


def test_binding_loads_library_and_sets_signatures(lib):
    from paper_1909_11474_gb300 import binding
    L = binding.load()
    assert L.tersoff_eval.restype is ctypes.c_int
    # null context is rejected on the host before any CUDA call
    assert L.tersoff_eval(None, None, 1, 32, None, None, None, None) == binding.E_ARG
    assert L.tersoff_last_error(None) == b""


def test_build_watches_every_included_file():
    """Each file that a source of the library includes is one whose change makes the objects stale."""
    from paper_1909_11474_gb300 import build
    deps = {os.path.realpath(d) for d in build._deps()}
    for name in os.listdir(build.CSRC):
        path = os.path.join(build.CSRC, name)
        for inc in re.findall(r'^\s*#include "([^"]+)"', open(path).read(), re.M):
            assert os.path.realpath(os.path.join(build.CSRC, inc)) in deps, f"{name} includes {inc}"


def test_current_stream_without_pytorchs_private_calls(monkeypatch):
    """The current stream's handle comes the public way where PyTorch has no private calls for it."""
    import types

    import torch

    from paper_1909_11474_gb300 import binding
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    monkeypatch.setattr(binding, "_raw_device", lambda: 3)
    monkeypatch.setattr(binding, "_raw_stream", lambda device: 100 + device)
    assert binding._stream(None) == 103
    monkeypatch.setattr(binding, "_raw_stream", None)
    assert binding._stream(None) == 1234
