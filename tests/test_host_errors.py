"""The library's host code with a fake of the CUDA runtime (host_fake.cpp): a
launch that fails leaves nothing behind on the tree's second stream that the
caller's stream does not wait for; the monopole weights' table is exact."""

import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1908_03121_gb300", "csrc")


def _program(tmp_path):
    cc = shutil.which("g++")
    include = "/usr/local/cuda/include"
    if cc is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = tmp_path / "host"
    subprocess.run([cc, "-std=c++17", "-O1", "-I" + include, "-I" + CSRC, os.path.join(CSRC, "fmm_host.cpp"),
                    os.path.join(HERE, "host_fake.cpp"), "-o", str(exe)], check=True)
    return str(exe)


def test_streams_are_joined_after_a_failed_launch(tmp_path):
    r = subprocess.run([_program(tmp_path)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("theta", [0.577, 0.5, 0.28])
def test_monopole_weights_are_correctly_rounded(tmp_path, theta):
    """The transformed weights against exact sums: the same table on every host."""
    r = subprocess.run([_program(tmp_path), str(theta)], capture_output=True, text=True, timeout=60, check=True)
    out = r.stdout.split()
    n = int(out[0])
    orbits = np.array(out[1:1 + 4 * n], dtype=int).reshape(n, 4)
    coef = [float.fromhex(v) for v in out[1 + 4 * n:]]
    at = 0
    for dx, dy, dz, mask in orbits:
        w = np.empty((8, 8, 4), object)
        for p in range(8):
            for q in range(8):
                o = [2 * d + ((q >> i) & 1) - ((p >> i) & 1) for i, d in enumerate((dx, dy, dz))]
                r2 = float(sum(x * x for x in o))
                r = math.sqrt(r2)
                ir3 = 1.0 / (r2 * r)
                w[p, q] = [Fraction(float(v)) for v in (-1.0 / r, -o[0] * ir3, -o[1] * ir3, -o[2] * ir3)]
        for axis in (0, 1):
            w = np.moveaxis(w, axis, 0)
            for bit in (1, 2, 4):
                keep = [w[i] for i in range(8)]
                w = np.array([keep[i & ~bit] + (-1 if i & bit else 1) * keep[i | bit] for i in range(8)])
            w = np.moveaxis(w, 0, axis)
        for b in range(8):
            for q in range(8):
                if q & ~mask:
                    continue
                for c in range(4):
                    a = q ^ b ^ (0 if c == 0 else 1 << (c - 1))
                    assert coef[at] == float(w[a, b, c] / 64), (dx, dy, dz, a, b, c)
                    at += 1
    assert at == len(coef) - 8
