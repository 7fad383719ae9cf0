"""How the binding's native module is built, and what the binding hands to it."""
from __future__ import annotations

import ctypes
import subprocess
import sys

import pytest
import torch

from paper_2604_00529_b200 import binding, build


def test_one_cpp_runtime_in_the_process():
    """The module exchanges strings, streams and exceptions with torch, so it takes the process's C++ runtime."""
    so = build.build_host_module()
    dynamic = subprocess.run(["readelf", "-d", so], capture_output=True, text=True, check=True).stdout
    assert "[libstdc++.so.6]" in dynamic and "[libtorch_python.so]" in dynamic


def test_prepared_calls_leave_other_arguments_to_the_call(monkeypatch):
    """What is no 64-bit integer is converted (a count beyond 2^63 modulo 2^64) or refused when the call is made."""
    seen = []
    fn = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)(
        lambda *a: seen.append(a) or 0)
    monkeypatch.setattr(binding, "_stream", lambda stream: 9)
    binding.PreparedCall(fn, (64, 1, 2 ** 64 - 32, 128), "mxq_fake_quant_bwd", ())()
    assert seen == [(64, 1, 2 ** 64 - 32, 128, 9)]
    refused = binding.PreparedCall(fn, (64, 1, 32.0, 128), "mxq_fake_quant_bwd", ())
    with pytest.raises(ctypes.ArgumentError):
        refused()


def test_each_torch_and_python_has_a_module_of_its_own(monkeypatch):
    built = build.host_module_path()
    for target, name, value in ((torch, "__version__", "99.1.0+cu999"), (build.sysconfig, "get_config_var", lambda v: ".cpython-399.so")):
        with monkeypatch.context() as m:
            m.setattr(target, name, value)
            assert build.host_module_path() != built and not build.os.path.exists(build.host_module_path())
            m.setattr(binding, "_lib", None)
            m.setattr(binding, "_host", None)
            with pytest.raises(ImportError, match="not built"):
                binding.load_library()
    assert build.host_module_path() == built and binding.load_library() is not None


def test_the_c_library_builds_without_torch(monkeypatch, tmp_path, capsys):
    built = []
    monkeypatch.setattr(build, "_build_library", lambda *a, **k: built.append(a) or "libmxq.so")
    (tmp_path / "torch").mkdir()
    with monkeypatch.context() as m:
        m.setattr(torch, "__file__", str(tmp_path / "torch" / "__init__.py"))        # a torch without CUDA libraries
        assert build.build() == "libmxq.so"
    with monkeypatch.context() as m:
        m.setitem(sys.modules, "torch", None)                                        # none at all
        assert build.build() == "libmxq.so"
    assert len(built) == 2 and capsys.readouterr().err.count("_mxq_host is not") == 2
