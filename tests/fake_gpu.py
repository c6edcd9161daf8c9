"""Runs a piece of Python against libwf.so on the runtime of fake_cudart.cpp,
in a process of its own: for what the library asks of the CUDA runtime on
devices, or in orders of calls, that a machine with one GPU cannot show."""

import os
import shutil
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, os, sys
sys.path.insert(0, {root!r})
import numpy as np
from paper_1704_00865_gb300 import synth, wf
lib, fake = wf.load(), C.CDLL({so!r})
fake.fake_alloc.restype, fake.fake_alloc.argtypes = C.c_void_p, [C.c_size_t]
fake.fake_launch.restype = C.c_char_p
NO_STREAM = C.c_void_p(None)

def launches(first=0):
    '''[(device, kernel, dynamic shared memory, refused)] from launch `first` on'''
    out = []
    for i in range(first, fake.fake_launches()):
        d, s, r = C.c_int(), C.c_size_t(), C.c_int()
        name = fake.fake_launch(i, C.byref(d), C.byref(s), C.byref(r))
        out.append((d.value, name.decode(), s.value, bool(r.value)))
    return out
"""


def run(tmp_path, body):
    """Run `body` after the prelude; fails with the process's output."""
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if cxx is None or not os.path.exists(nvcc):
        pytest.skip("no host C++ compiler or no CUDA headers")
    from paper_1704_00865_gb300 import build
    build.build()
    so = str(tmp_path / "fake_cudart.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, os.path.join(HERE, "fake_cudart.cpp"),
                        "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    code = PRELUDE.format(root=ROOT, so=so) + textwrap.dedent(body)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=so))
    assert r.returncode == 0, r.stdout + r.stderr
