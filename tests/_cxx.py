"""Test helper: compile a C++ program against the library's internal headers (and
the library) with g++ and run it.  No GPU is used."""
import os
import shutil
import subprocess

import pytest

from _lib import tnlib


def run_cxx(tmp_path, source, link=True):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    tnlib()
    from paper_2110_14502_gb300 import build as B
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(source)
    cmd = [gxx, "-std=c++17", "-O1", "-pthread", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), "-I", cuda, src,
           "-o", exe]
    if link:
        cmd += ["-L", B.PKG, "-ltn", f"-Wl,-rpath,{B.PKG}"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
