"""The evaluation driver (csrc/api.cpp) checked as plain C++ on a stand-in device (host_eval_check.cpp): without
room for the streaming greedy's buffers a set of patterns is cut for the windowed rounds and evaluated whole."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

from .test_host_checks import CSRC, ROOT


def test_no_room_for_the_streaming_buffers(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.path.join(os.environ.get("CUDA_HOME") or "/usr/local/cuda", "include")
    if not cxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-isystem", cuda,
                    os.path.join(ROOT, "tests", "host_eval_check.cpp"),
                    *[os.path.join(CSRC, s) for s in ("api.cpp", "graph.cpp", "pattern.cpp")], "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "fails 0" in r.stdout, r.stdout + r.stderr
