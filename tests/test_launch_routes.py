"""Which kernels the library's calls launch, checked without a GPU: its objects
linked against a stand-in for the CUDA runtime (launch_routes.cpp)."""
import importlib
import os
import subprocess

import pytest

import paper_2311_03694_gb300 as grom
from test_plan_invariants import _cuda_include

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
grom_build = importlib.import_module("paper_2311_03694_gb300.build")  # the package's `build` is its function


def test_launch_routes(tmp_path):
    grom.build()
    inc = _cuda_include()
    objs = [os.path.join(grom_build.BUILD, os.path.splitext(s)[0] + ".o") for s in grom_build.SOURCES]
    if inc is None or not all(os.path.exists(o) for o in objs):
        pytest.skip("CUDA headers or the library's objects not found")
    exe = str(tmp_path / "launch_routes")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + inc, "-I" + os.path.join(ROOT, "include"),
                    os.path.join(HERE, "launch_routes.cpp")] + objs + ["-lpthread", "-ldl", "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and ", 0 failed" in r.stdout, r.stdout[-3000:] + r.stderr[-1000:]
