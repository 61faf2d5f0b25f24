"""Compiles a C++ test program of the library's host code (tests/host) against fakes of
the CUDA calls it makes, and runs it: what the code does when a call fails, or with
memory that only CUDA may touch, without a GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1109_3266_gb300", "csrc")


def program(tmp_path_factory, name, *library_sources):
    """The built test program tests/host/<name>.cpp with the given sources of the library."""
    from paper_1109_3266_gb300 import build
    try:
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    except RuntimeError:
        pytest.skip("no CUDA headers")
    out = str(tmp_path_factory.mktemp(name) / name)
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-pthread", "-I", SRC, "-I", build.INCLUDE, "-I", cuda,
           os.path.join(ROOT, "tests", "host", name + ".cpp")]
    for s in library_sources:
        cmd += ["-x", "c++", os.path.join(SRC, s)]
    r = subprocess.run(cmd + ["-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def run(prog, *args):
    r = subprocess.run([prog, *map(str, args)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout + r.stderr)
    return r.stdout
