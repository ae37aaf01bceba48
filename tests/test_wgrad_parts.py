"""The split of a weight gradient's batch rows over CTAs (wgrad_parts in
csrc/rlt2_mlp_gemm.h), compiled for the host: a tensor-core accumulator's error
grows with the rows that it sums, so no part holds more than 1,024 rows (512 up to
32,768 rows) beyond the rounding up to whole 64-row steps, whatever the width, the
batch and the SM count; parts stay above one step."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_1710_03732_gb300", "csrc")
SHIM = r"""
#include "rlt2_mlp_gemm.h"
extern "C" int parts(int K, int blocks, int sms) { return rlt2::wgrad_parts(K, blocks, sms); }
"""


@pytest.fixture(scope="module")
def parts(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("parts")
    src, so = d / "shim.cpp", d / "libparts.so"
    src.write_text(SHIM)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + HDR,
                        "-I" + os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include"), str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so)).parts


@pytest.mark.parametrize("blocks", [1, 2, 4, 8, 200])
@pytest.mark.parametrize("sms", [1, 76, 148, 152])
def test_rows_of_a_part_are_bounded(parts, blocks, sms):
    for K in list(range(64, 9000, 64)) + list(range(9024, 262144 + 64, 1088)) + [32704, 32768, 32832, 65536, 262144]:
        p = parts(K, blocks, sms)
        assert p >= 1
        if K < 2048:
            assert p == 1
            continue
        # rows of one part as umma_gemm cuts them: whole steps of 64
        rows = -(-(K // p) // 64) * 64
        assert rows <= (512 if K <= 32768 else 1024) + 64, (K, p)
        assert K // p >= 256, (K, p)
