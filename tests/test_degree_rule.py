"""Which steps are laid out by degree (csrc/layout.h): the CSR kernels that walk rows, except the staged
stream and the looped persistent form; not the atomic scatter."""
import os
import shutil
import subprocess

import pytest

from paper_1911_10274_gb300 import titan as T

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")


def test_rule(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    want = [(T.ACCUM_CSR, v, loop, v != 2 and not loop) for v in range(9) for loop in (False, True)]
    want += [(T.ACCUM_ATOMIC, v, loop, False) for v in range(9) for loop in (False, True)]
    src = tmp_path / "t.cpp"
    src.write_text('#include "layout.h"\n' + "".join(
        f"static_assert(titan::degree_order_helps({a}, {v}, {str(p).lower()}) == {str(w).lower()}, \"\");\n"
        for a, v, p, w in want) + """using namespace titan;
static_assert(may_run_looped(4096, TITAN_EXEC_AUTO, true) && may_run_looped(1, TITAN_EXEC_PERSISTENT, true), "");
static_assert(!may_run_looped(4097, TITAN_EXEC_AUTO, true) && !may_run_looped(9, TITAN_EXEC_AUTO, false), "");
static_assert(!may_run_looped(9, TITAN_EXEC_LAUNCH, true), "");
""")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-c", str(src), "-o",
                    str(tmp_path / "t.o")], check=True)


def test_create_asks_the_rule():
    text = open(os.path.join(CSRC, "runtime.cu")).read()
    at = text.index("titan::degree_order(")
    assert "if (titan::degree_order_helps(p->accumulate, p->kernel_variant, titan::may_run_looped(" in text[at - 200:at]
    assert text.count("degree_order(") == 1
