"""Host plan of the row-register batch form: a CTA holds up to 384 masses of actuated batches and up to 512 of
unactuated ones - what an SM's registers hold of each - so that systems take the fewest CTAs."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from test_batch_rows_host import CSRC, ROOT, lib  # noqa: F401
from test_gpu_batch_rows import _box

# what an SM holds of either: 512-thread CTAs at 128 registers, 384 at 168
SIZES = [(8, 8, 6), (11, 7, 5), (8, 8, 8), (9, 19, 3), (16, 8, 8), (12, 12, 12)]


@pytest.mark.parametrize("act,want", [(True, [1, 2, 2, 2, 3, 5]), (False, [1, 1, 1, 2, 2, 4])], ids=["actuated", "plain"])
def test_ctas_per_system(lib, act, want, tmp_path):  # noqa: F811
    from paper_1911_10274_gb300 import titan as T
    (tmp_path / "c.cpp").write_text("""#include "layout.h"
using namespace titan;
extern "C" int clusters(unsigned n, const titan_masses *m, const titan_springs *s, const titan_actuation *a, unsigned *cl,
                        unsigned *threads) {
    BatchHost L;
    std::string why;
    BatchPlan plan;
    plan.rows = true;
    if (!build_batch(n, m, s, a, L, &why, plan)) return 1;
    for (const BatchGroup &g : L.groups)
        for (unsigned c = g.cta_first; c < g.cta_first + g.cta_count; ++c) {
            cl[L.ctas[c].robot] = g.cluster;
            threads[L.ctas[c].robot] = g.row_threads;
        }
    return 0;
}
""")
    so = str(tmp_path / "c.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(CSRC, "layout.cpp"), str(tmp_path / "c.cpp"), "-o", so], check=True)
    keep, ms, ss, acts = [], [], [], []
    for k, size in enumerate(SIZES):
        sy = _box(*size, k, act)
        d = [np.ascontiguousarray(x, t) for x, t in ((sy.pos, np.float64), (sy.vel, np.float64), (sy.mass, np.float64),
                                                     (sy.fixed, np.uint8), (sy.ends, np.uint32), (sy.k, np.float64),
                                                     (sy.rest, np.float64))]
        if act:
            d += [np.ascontiguousarray(sy.act_amp, np.float64), np.ascontiguousarray(sy.act_phase, np.float64)]
        p = [x.ctypes.data for x in d]
        keep.append(d)
        ms.append(T.titan_masses(sy.n_masses, *p[:4]))
        ss.append(T.titan_springs(sy.n_springs, *p[4:7], None))
        acts.append(T.titan_actuation(p[7], p[8], 2.0) if act else T.titan_actuation(None, None, 0.0))
    n = len(ms)
    cl, th = (C.c_uint32 * n)(), (C.c_uint32 * n)()
    M, S, A = (T.titan_masses * n)(*ms), (T.titan_springs * n)(*ss), (T.titan_actuation * n)(*acts)
    assert C.CDLL(so).clusters(n, M, S, A, cl, th) == 0
    assert list(cl) == want
    assert max(th) <= (384 if act else 512)
    if act:                                       # and the plan holds together
        assert lib.check(n, M, S, A, (C.c_uint32 * n)()) == 0
