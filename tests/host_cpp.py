"""Compiles a C++ program against the library's CUDA-free headers (csrc/*.h) and returns what it prints."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_07929_gb300", "csrc")


def run(source: str, tmp_path, stdin: str = "") -> str:
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = os.path.join(tmp_path, "prog.cc"), os.path.join(tmp_path, "prog")
    with open(src, "w") as f:
        f.write(source)
    res = subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, "-o", exe, src], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return subprocess.run([exe], input=stdin, capture_output=True, text=True, check=True, timeout=60).stdout
