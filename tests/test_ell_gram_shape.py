"""The launch of the sparse FP32 product that also sums P^T A P and P^T r: a
lane meets one row per slice of its warp and adds their products in FP32, at
most 64 of them before the sums leave the lane, whatever the matrix.  The rule
runs as host code on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path_factory.mktemp("ell") / "ell_gram_check")
    csrc = os.path.join(ROOT, "paper_2402_12833_gb300", "csrc")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "native", "ell_gram_check.cpp"), "-o", exe], check=True)

    def run(nslices, sms):
        out = subprocess.run([exe, str(nslices), str(sms)], check=True, capture_output=True, text=True).stdout
        return tuple(int(v) for v in out.split())
    return run


@pytest.mark.parametrize("sms", [1, 152])
@pytest.mark.parametrize("nslices", [1, 7, 8, 9, 8 * 152 * 8, 8 * 152 * 8 * 64, 8 * 152 * 8 * 64 + 1,
                                     30_000_000 // 32, 30_000_000 // 8, 2 ** 31 // 32])
def test_a_lane_sums_at_most_64_rows(check, nslices, sms):
    blocks, slices = check(nslices, sms)
    assert slices <= 64
    assert 1 <= blocks <= -(-nslices // 8)             # no block without a slice
    if nslices <= 8 * sms * 8 * 64:                    # within the limit: eight blocks per SM at most
        assert blocks <= 8 * sms
