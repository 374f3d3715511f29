"""What is kept per CUDA context (csrc/context_id.h) is used again in that context only: not in another, and
not where the driver gives no id; the two places that keep something ask there."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_10274_gb300", "csrc")


def test_same_context(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text('#include "context_id.h"\nusing titan::same_context;\n'
                   "static_assert(same_context(7, 7) && !same_context(7, 8) && !same_context(7, 0) && "
                   "!same_context(0, 7) && !same_context(0, 0), \"\");\nint main() {}\n")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-c", str(src), "-o", str(tmp_path / "t.o")], check=True)


@pytest.mark.parametrize("name", ["adjoint.cu", "noalloc.cu"])
def test_kept_ids_are_compared_there(name):
    text = open(os.path.join(CSRC, name)).read()
    assert "same_context(" in text and "ctx_id ==" not in text and "ctx_id !=" not in text
