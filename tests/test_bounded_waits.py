"""Device-side waits give up after about a second and say so by their result.  A kernel that does not look at it goes on with
operands that never came: no call may drop the result."""
import os
import re
import subprocess

import pytest

from paper_2509_24695_b200 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")
SOURCES = sorted(os.path.basename(f) for f in build.sources())


def dropped(text):
    """Lines on which a call of mbar_wait is a statement of its own."""
    text = re.sub(r"//[^\n]*", "", text)
    return [text.count("\n", 0, m.start()) + 1 for m in re.finditer(r"\bmbar_wait\s*\(", text) if text[:m.start()].rstrip()[-1] in ";{})"]


def test_the_check_sees_a_dropped_result():
    assert len(dropped("if (t) mbar_wait(a, 0, f);")) == 1 and len(dropped("x = 1;\n  mbar_wait(a, 0, f);")) == 1
    assert not dropped("if (!mbar_wait(a, 0, f)) break; ok = mbar_wait(b, 1, f); __all_sync(m, mbar_wait(c, 1, f));")


@pytest.mark.parametrize("name", SOURCES)
def test_no_result_is_dropped(name):
    lines = dropped(open(os.path.join(CSRC, name)).read())
    assert not lines, f"{name}: a wait's result is dropped on lines {lines}"


@pytest.mark.parametrize("statement,compiles", [("if (!mbar_wait(b, 0, f)) return;", True), ("mbar_wait(b, 0, f);", False)])
def test_the_build_refuses_a_dropped_result(tmp_path, statement, compiles):
    src = tmp_path / "t.cu"
    src.write_text('#include "sm100_ptx.cuh"\n__global__ void t(uint64_t* b, volatile int* f) { using namespace linattn::ptx; %s }\n' % statement)
    rc = subprocess.run(["nvcc", *build.NVCC_FLAGS, "-I", CSRC, "-c", str(src), "-o", str(tmp_path / "t.o")], capture_output=True).returncode
    assert (rc == 0) == compiles
