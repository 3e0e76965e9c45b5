"""The root and the reciprocal of the step: FP32 rounds as CUDA's (two steps per launch give the
bits of single steps), from any approximation within two units; FP64 is within a unit."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1708_07525_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def library(cmd, tmp_path, source):
    path = str(tmp_path / "roots.so")
    r = subprocess.run(cmd + ["-I", build.CSRC, "-shared", "-o", path, os.path.join(HERE, source)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(path)


def test_sequences_round_as_the_exact_result_does(tmp_path):
    L = library(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC"], tmp_path, "roots_host.cpp")
    wrong = (C.c_longlong * 2)()
    L.check_roots(2, wrong)
    assert list(wrong) == [0, 0]


@pytest.mark.gpu
def test_roots_on_the_gpu(tmp_path):
    L = library([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-cudart", "static"],
                tmp_path, "roots_gpu.cu")
    out = (C.c_ulonglong * 6)()
    assert L.check_roots(out) == 0
    assert list(out)[:2] == [0, 0]
    # the series' next term is below 2^-57 for seeds within 2^-19; x y is rounded once before it
    # (half a unit at most), the result once
    assert out[2] <= 1 and out[3] <= 1
    assert out[4] < 2 ** 11 and out[5] < 2 ** 11
