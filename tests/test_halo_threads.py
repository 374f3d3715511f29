"""build_halo (csrc/layout.cpp) with an allocation of the calling thread refused, each of the first ones in
turn: among them those that start its threads.  It gives the same tables or throws bad_alloc; the process goes
on."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include <random>
#include "layout.h"
static thread_local long left = -1;             // allocations of this thread until one is refused (-1: none)
static bool refused = false;
void *operator new(size_t n) {
    if (left > 0 && --left == 0) { left = -1; refused = true; throw std::bad_alloc(); }
    void *p = malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
int main() {
    using namespace titan;
    const uint32_t n = 256 * 70, s = 3 * n;
    std::mt19937 rng(1);
    std::vector<uint32_t> ends, dev(n);
    std::vector<double> pos(3 * n);
    for (auto &x : pos) x = rng() / 4294967296.0;
    for (uint32_t i = 0; i < n; ++i) dev[i] = i;
    for (uint32_t q = 0; q < s; ++q) {
        const uint32_t a = rng() % n;
        ends.push_back(a);
        ends.push_back((a + 1 + rng() % 300) % n);
    }
    SellHost sell;
    if (!build_sell(n, s, ends.data(), pos.data(), dev, sell)) return 2;
    HaloHost want, got;
    if (!build_halo(n, sell, 4096, false, want)) return 3;
    int thrown = 0, whole = 0;
    for (long k = 1; k <= 60; ++k) {
        got = HaloHost();
        refused = false;
        left = k;
        try {
            if (!build_halo(n, sell, 4096, false, got)) return 4;
            left = -1;
            if (got.ext_idx != want.ext_idx || got.ext_off != want.ext_off || got.ext_slot != want.ext_slot ||
                got.nbr_slot != want.nbr_slot || got.own_slot != want.own_slot || got.max_table != want.max_table)
                return 5;
            whole += refused;
        } catch (const std::bad_alloc &) {
            left = -1;
            ++thrown;
        }
    }
    printf("%d refusals thrown, %d survived\n", thrown, whole);
    return thrown && whole ? 0 : 6;
}
"""


def test_refused_allocations(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    if (os.cpu_count() or 1) < 3:
        pytest.skip("needs several host threads")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(CSRC, "layout.cpp"), str(tmp_path / "main.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
