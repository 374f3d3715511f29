"""Which shapes go to the CTA-pair product (csrc/gemm_rule.h): the shapes that test_gpu_gemm_pairs_taken
multiplies do, and on 152 SMs the lines lie where the measurements put them."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

from test_gpu_gemm_pairs_taken import SHAPES

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_10274_gb300", "csrc")


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rule")
    (d / "r.cpp").write_text('#include "gemm_rule.h"\nextern "C" int pairs(long M, long N, long K, int sms) '
                             "{ return titan::gemm_takes_pairs(M, N, K, sms); }\n"
                             'extern "C" int width(long M, long N, long K, int gelu) '
                             "{ return titan::gemm_tile_width(M, N, K, gelu); }\n")
    out = str(d / "r.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cpp"), "-o", out], check=True)
    lib = C.CDLL(out)
    for fn in (lib.pairs, lib.width):
        fn.argtypes = [C.c_long] * 3 + [C.c_int]
    return lib


@pytest.fixture
def pairs(rules):
    return lambda M, N, K, sms=152: bool(rules.pairs(M, N, K, sms))


def test_tested_shapes_take_pairs(pairs):
    assert all(pairs(*s) for s in SHAPES)


@pytest.mark.parametrize("M,N,K,want", [
    (20 * 256, 19 * 256, 64, True), (20 * 256, 18 * 256, 64, False),          # 380 tiles: five a pair
    (8 * 256, 19 * 256, 512, True), (8 * 256, 19 * 256, 448, False),          # 152: two a pair, K from 512
    (5 * 256, 19 * 256, 1024, True), (5 * 256, 19 * 256, 960, False),         # 95: five quarters, K from 1024
    (2 * 256, 47 * 256, 4096, False), (4 * 256, 19 * 256, 8192, True),        # 94; 76: one a pair, K from 8192
    (4 * 256, 19 * 256, 8128, False), (3 * 256, 25 * 256, 1 << 16, False),    # 75: not every pair has one
    (32 * 256 + 128, 32 * 256, 8192, False), (32 * 256, 32 * 256 + 128, 8192, False), (8192, 8192, 8192, True)])
def test_lines(pairs, M, N, K, want):
    assert pairs(M, N, K) == want


@pytest.mark.parametrize("M,N,K,gelu,want", [
    (1024, 512, 1024, True, 64), (128 * 38, 512, 512, True, 64), (128 * 39, 512, 512, True, 128),    # 152, 156 tiles
    (32768, 512, 512, True, 128), (32768, 512, 512, False, 256), (16384, 4096, 4096, True, 256),
    (16384, 4096, 4032, True, 128), (128 * 19, 4096, 4096, True, 256), (128 * 18, 4096, 4096, True, 128),   # 304, 288
    (16384, 4096 + 128, 4096, True, 128), (16384, 4096 + 128, 4096, False, 128)])
def test_tile_width(rules, M, N, K, gelu, want):
    assert rules.width(M, N, K, gelu) == want
