"""The library's host code with a fake of the CUDA runtime (host_fake.cpp): a
launch that fails leaves nothing behind on the tree's second stream that the
caller's stream does not wait for."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1908_03121_gb300", "csrc")


def test_streams_are_joined_after_a_failed_launch(tmp_path):
    cc = shutil.which("g++")
    include = "/usr/local/cuda/include"
    if cc is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = tmp_path / "host"
    subprocess.run([cc, "-std=c++17", "-O1", "-I" + include, "-I" + CSRC, os.path.join(CSRC, "fmm_host.cpp"),
                    os.path.join(HERE, "host_fake.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
