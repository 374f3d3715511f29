"""Parameter offsets and gradient indexes of the surrogate (csrc/mlp_layout.h) against whole numbers of
any size, for ordinary networks and for ones of more than 2^32 parameters, or weights in one layer."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")
SHIM = """#include "mlp_layout.h"
using namespace titan;
extern "C" void layout(unsigned in, unsigned hid, unsigned long long *o) {
    const MlpLayout m = mlp_layout(in, hid);
    for (int l = 0; l < 3; ++l) { *o++ = m.w[l]; *o++ = m.n_w[l]; *o++ = m.b[l]; }
    *o++ = m.w4; *o++ = m.b4; *o++ = m.total;
    for (int l = 0; l < 3; ++l) { *o++ = grad_blocks(m.n_w[l]); *o++ = grad_index(grad_blocks(m.n_w[l]) - 1, 255); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("mlp_layout")
    (d / "shim.cpp").write_text(SHIM)
    out = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", out], check=True)
    return C.CDLL(out)


@pytest.mark.parametrize("n_in,hidden", [(128, 128), (1024, 512), (128, 46464), (46464, 46464), (128, 65536), (128, 79872)])
def test_layout(lib, n_in, hidden):
    got = (C.c_ulonglong * 18)()
    lib.layout(n_in, hidden, got)
    want, at = [], 0
    for n in (n_in * hidden, hidden * hidden, hidden * hidden):
        want += [at, n, at + n]
        at += n + hidden
    want += [at, at + hidden, at + hidden + 1]
    for n in (n_in * hidden, hidden * hidden, hidden * hidden):
        want += [n // 1024, n - 4]            # the last thread forms the last four weights
    assert list(got) == want
