"""How persistent systems are planned (csrc/layout.h): which run in the row-register form, and for how many
masses a CTA."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_10274_gb300", "csrc")
RULES = """#include "layout.h"
using namespace titan;
// masses, per-spring damping, actuated, sinusoid
static_assert(persist_aim(27, false, false, true) == 512 && persist_aim(27, false, true, false) == 384, "");
static_assert(persist_aim(255, false, true, true) == 512 && persist_aim(256, false, true, true) == 384, "");
static_assert(persist_aim(500, true, true, false) == 512 && persist_aim(500, true, false, true) == 512, "");
static_assert(!persist_rows_wanted(500, true, false, true) && persist_rows_wanted(27, false, false, true), "");
"""


def test_rules(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    (tmp_path / "t.cpp").write_text(RULES)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-c", str(tmp_path / "t.cpp"),
                    "-o", str(tmp_path / "t.o")], check=True)
