"""component_order (csrc/layout.cpp): connected components get consecutive device indices, in the
order they are first met, each one's masses in their given order."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1911_10274_gb300 import inputs
from paper_1911_10274_gb300.titan import union_system

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")
SHIM = """#include "layout.h"
#include <cstring>
extern "C" void order(const double *pos, unsigned n, unsigned s, const unsigned *ends, unsigned *before, unsigned *after) {
    std::vector<unsigned> o;
    titan::morton_order(pos, n, o);
    memcpy(before, o.data(), 4 * n);
    titan::component_order(n, s, ends, o);
    memcpy(after, o.data(), 4 * n);
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    src, out = str(d / "order.cpp"), str(d / "liborder.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([shutil.which("g++"), "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(CSRC, "layout.cpp"), src, "-o", out], check=True)
    lib = C.CDLL(out)

    def call(pos, ends):
        pos, ends = np.ascontiguousarray(pos, np.float64), np.ascontiguousarray(ends, np.uint32)
        a, b = np.empty(len(pos), np.uint32), np.empty(len(pos), np.uint32)
        lib.order(pos.ctypes.data_as(C.c_void_p), len(pos), len(ends), ends.ctypes.data_as(C.c_void_p),
                  a.ctypes.data_as(C.c_void_p), b.ctypes.data_as(C.c_void_p))
        return a, b
    return call


def _by_hand(order, ends):
    label = np.arange(len(order))
    for _ in range(len(order)):                       # smallest label of the component, by relaxation
        new = label.copy()
        np.minimum.at(new, ends[:, 0], label[ends[:, 1]])
        np.minimum.at(new, ends[:, 1], label[ends[:, 0]])
        if np.array_equal(new, label):
            break
        label = new
    met, out = [], []
    for i in order:
        if label[i] not in met:
            met.append(label[i])
    for m in met:
        out += [i for i in order if label[i] == m]
    return np.array(out)


def test_overlapping_bodies_become_consecutive(order):
    rng = np.random.default_rng(0)
    sy, mo, _ = union_system([inputs.actuated_box(a, b, c, rng) for a, b, c in [(4, 3, 3), (2, 2, 2), (3, 5, 2)]])
    before, after = order(sy.pos, sy.ends)
    np.testing.assert_array_equal(after, _by_hand(before, sy.ends.astype(np.int64)))
    robot = np.searchsorted(mo, after, side="right")
    assert (np.diff(robot) != 0).sum() == 2 and (np.diff(np.searchsorted(mo, before, side="right")) != 0).sum() > 2


def test_single_masses_chains_and_one_component(order):
    rng = np.random.default_rng(1)
    pos = rng.uniform(size=(60, 3))
    ends = np.array([(i, i + 3) for i in range(0, 40)] + [(50, 45), (45, 59)])
    before, after = order(pos, ends)
    np.testing.assert_array_equal(after, _by_hand(before, ends))
    chain = np.stack([np.arange(59), np.arange(1, 60)], axis=1)
    before, after = order(pos, chain)
    np.testing.assert_array_equal(after, before)
