"""Host-side checks of the multi-right-hand-side application's launch geometry and
of the rule that chooses it, and of the wide bases' geometries
(paper_1608_04607_gb300/csrc/launch_geometry.h, shared with the CUDA code).
Compiles small C++ programs; no GPU needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("name", ["multi_geometry_check", "wide_geometry_check"])
def test_geometry(name):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out_dir = os.path.join(ROOT, "tests", "_build")
    os.makedirs(out_dir, exist_ok=True)
    exe = os.path.join(out_dir, name)
    src = os.path.join(ROOT, "tests", name + ".cpp")
    inc = os.path.join(ROOT, "paper_1608_04607_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", inc, src, "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.startswith("ok")
