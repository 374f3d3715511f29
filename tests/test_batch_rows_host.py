"""Host plan of the row-register batch form (build_batch with plan.rows): CTA
sizes, row widths, shared memory, and the copy lists - every halo entry of every
CTA is written by exactly the mass it copies, and by nothing else."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")

CHECK = r"""
#include <cstdio>
#include <map>
#include "layout.h"
using namespace titan;
// 0: every condition holds; else the number of the first that fails
extern "C" int check(uint32_t n, const titan_masses *m, const titan_springs *s, const titan_actuation *a, uint32_t *clusters) {
    BatchHost L;
    std::string why;
    BatchPlan plan;
    plan.rows = true;
    if (!build_batch(n, m, s, a, L, &why, plan)) return 1;
    for (const BatchGroup &g : L.groups) {
        if (!g.row_threads) return 2;
        if (g.row_threads > kRowSlots || g.smem > kBatchSmemLimit || g.cta_count % g.cluster) return 3;
        for (uint32_t c0 = g.cta_first; c0 < g.cta_first + g.cta_count; c0 += g.cluster) {
            clusters[L.ctas[c0].robot] = g.cluster;
            std::map<uint32_t, int> wrote;         // rank << 16 | halo entry -> times written
            for (uint32_t q = 0; q < g.cluster; ++q) {
                const BatchCta &d = L.ctas[c0 + q];
                const BatchSmem B = batch_smem_layout(d.slot_count, d.halo_slots, d.n_slices, d.edge_count, L.any_act);
                if (d.slot_count > g.row_threads || B.inv > g.row_smem || d.halo_count > d.halo_slots) return 4;
                for (uint32_t i = 0; i < d.n_slices; ++i)
                    if ((L.slices[d.slice_base + i + 1] - L.slices[d.slice_base + i]) / 32 > kRowWidth) return 5;
                for (uint32_t h = 0; h < d.halo_count; ++h) {       // the halo's initial state is read from here
                    const uint32_t code = L.halo[d.halo_off + h], o = code >> 16, sl = code & 0xffff;
                    if (o >= g.cluster || sl >= L.ctas[c0 + o].mass_count) return 6;
                    if (d.mass_begin + (int)(o - q) * (int)d.slot_count + sl != L.ctas[c0 + o].mass_begin + sl) return 7;
                }
                if (g.cluster == 1) continue;
                for (uint32_t k = 0; k < d.mass_count; ++k) {
                    const uint32_t *pc = &L.push[2 * (size_t)(d.mass_begin + k)];
                    std::vector<uint32_t> to;
                    if (pc[0] != kNoPush) to.push_back(pc[0]);
                    if (pc[1] != kNoPush) {
                        if (pc[0] == kNoPush) return 8;
                        if (pc[1] & kMorePush) {
                            const uint32_t at = pc[1] & ~kMorePush;
                            if (at >= L.push_more.size() || at + L.push_more[at] >= L.push_more.size()) return 9;
                            for (uint32_t x = 1; x <= L.push_more[at]; ++x) to.push_back(L.push_more[at + x]);
                        } else to.push_back(pc[1]);
                    }
                    for (uint32_t code : to) {
                        const uint32_t r = code >> 16, h = code & 0xffff;
                        if (r >= g.cluster || r == q || h >= L.ctas[c0 + r].halo_count) return 10;
                        if (L.halo[L.ctas[c0 + r].halo_off + h] != (q << 16 | k)) return 11;
                        ++wrote[code];
                    }
                }
            }
            size_t halos = 0;
            for (uint32_t q = 0; q < g.cluster; ++q) halos += L.ctas[c0 + q].halo_count;
            if (g.cluster > 1 && wrote.size() != halos) return 12;
            for (auto &w : wrote)
                if (w.second != 1) return 13;
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rows")
    (d / "check.cpp").write_text(CHECK)
    out = str(d / "check.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(CSRC, "layout.cpp"), str(d / "check.cpp"), "-o", out], check=True)
    return C.CDLL(out)


@pytest.mark.parametrize("name,want", [("one_warp", [1, 1]), ("last_slot_and_one_more", [1, 2]),
                                       ("clusters_2_3_4", [1, 2, 4]), ("clusters_5_6_8", [5, 6, 8]),
                                       ("many_copies", [3, 2])])
def test_row_plan(lib, name, want):
    from paper_1911_10274_gb300 import titan as T
    from test_gpu_batch_rows import CASES
    keep, ms, ss, acts = [], [], [], []
    for sy in CASES[name](True):
        d = [np.ascontiguousarray(x, t) for x, t in ((sy.pos, np.float64), (sy.vel, np.float64), (sy.mass, np.float64),
                                                     (sy.fixed, np.uint8), (sy.ends, np.uint32), (sy.k, np.float64),
                                                     (sy.rest, np.float64), (sy.act_amp, np.float64),
                                                     (sy.act_phase, np.float64))]
        p = [x.ctypes.data for x in d]
        keep.append(d)
        ms.append(T.titan_masses(sy.n_masses, *p[:4]))
        ss.append(T.titan_springs(sy.n_springs, *p[4:7], None))
        acts.append(T.titan_actuation(p[7], p[8], 2.0))
    n = len(ms)
    clusters = (C.c_uint32 * n)()
    rc = lib.check(n, (T.titan_masses * n)(*ms), (T.titan_springs * n)(*ss), (T.titan_actuation * n)(*acts), clusters)
    assert rc == 0, f"condition {rc}"
    assert list(clusters) == want
