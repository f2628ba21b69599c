"""No C++ exception crosses the C ABI, and a call that found no host memory leaves its context as it was
(tests/host_memory_main.cpp, an executable whose operator new fails on purpose)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_calls_without_host_memory(tmp_path):
    from paper_2011_00287_gb300 import build as B
    lib = B.build()
    exe = str(tmp_path / "host_memory")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I" + os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "host_memory_main.cpp"), "-o", exe, lib,
                    "-Wl,-rpath," + os.path.dirname(lib)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), (r.returncode, r.stdout, r.stderr)
