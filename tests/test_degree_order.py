"""degree_order (csrc/layout.cpp) permutes masses within blocks of 256 only, by decreasing degree and
stably, and build_sell with its rank keeps every mass's row in the order it had without it."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")
SHIM = """#include "layout.h"
#include <cstring>
static void rows(const double *pos, unsigned n, unsigned s, const unsigned *ends, const std::vector<unsigned> &o,
                 const unsigned *rank, unsigned *out, unsigned *entries) {
    std::vector<unsigned> dev(n);
    for (unsigned d = 0; d < n; ++d) dev[o[d]] = d;
    titan::SellHost sell;
    titan::build_sell(n, s, ends, pos, dev, sell, nullptr, rank);
    *entries = sell.entries;
    for (unsigned i = 0, k = 0; i < n; ++i) {          // springs of caller mass i, in row order
        const unsigned d = dev[i], e0 = sell.slice_off[d / 32], w = (sell.slice_off[d / 32 + 1] - e0) / 32;
        for (unsigned t = 0; t < w; ++t)
            if (sell.spring[e0 + 32 * t + d % 32] != 0xffffffffu) out[k++] = sell.spring[e0 + 32 * t + d % 32];
    }
}
extern "C" void order(const double *pos, unsigned n, unsigned s, const unsigned *ends, unsigned *before,
                      unsigned *after, unsigned *rank_out, unsigned *rows_before, unsigned *rows_after, unsigned *entries) {
    std::vector<unsigned> o, rank;
    titan::morton_order(pos, n, o);
    memcpy(before, o.data(), 4 * n);
    rows(pos, n, s, ends, o, nullptr, rows_before, entries);
    titan::degree_order(n, s, ends, o, rank);
    memcpy(after, o.data(), 4 * n);
    memcpy(rank_out, rank.data(), 4 * n);
    rows(pos, n, s, ends, o, rank.data(), rows_after, entries + 1);
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("degree")
    src, out = str(d / "order.cpp"), str(d / "liborder.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([shutil.which("g++"), "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), os.path.join(CSRC, "layout.cpp"), src, "-o", out], check=True)
    lib = C.CDLL(out)

    def call(pos, ends):
        pos, ends = np.ascontiguousarray(pos, np.float64), np.ascontiguousarray(ends, np.uint32)
        n, s = len(pos), len(ends)
        a = [np.empty(k, np.uint32) for k in (n, n, n, 2 * s, 2 * s, 2)]
        lib.order(pos.ctypes.data_as(C.c_void_p), n, s, ends.ctypes.data_as(C.c_void_p),
                  *(x.ctypes.data_as(C.c_void_p) for x in a))
        return a
    return call


@pytest.mark.parametrize("n", [1, 31, 256, 257, 3000])
def test_degree_order(order, n):
    rng = np.random.default_rng(n)
    pos = rng.uniform(size=(n, 3))
    ends = inputs.knn_pairs(pos, min(6, n - 1)) if n > 1 else np.empty((0, 2), np.uint32)
    deg = np.bincount(ends.astype(np.int64).ravel(), minlength=n)
    before, after, rank, rows0, rows1, entries = order(pos, ends)
    assert np.array_equal(after, before[rank])
    for b in range(0, n, 256):
        r = rank[b:b + 256]
        assert sorted(r.tolist()) == list(range(b, min(n, b + 256)))
        key = [(-deg[before[i]], i) for i in r]
        assert key == sorted(key)
    assert np.array_equal(rows0, rows1)                # every mass's springs, in the same order
    assert entries[1] <= entries[0]
