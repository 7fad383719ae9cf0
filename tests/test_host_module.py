"""How the binding's native module is built: what it links, and when it is built again."""
from __future__ import annotations

import subprocess

from paper_2604_00529_b200 import build


def test_one_cpp_runtime_in_the_process():
    """The module exchanges strings, streams and exceptions with torch, so it takes the process's C++ runtime."""
    so = build.build_host_module()
    dynamic = subprocess.run(["readelf", "-d", so], capture_output=True, text=True, check=True).stdout
    assert "[libstdc++.so.6]" in dynamic and "[libtorch_python.so]" in dynamic
