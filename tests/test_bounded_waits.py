"""Device-side waits give up after about a second and say so by their result.  A kernel that does not look at it goes on with
operands that never came: no call may drop the result."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")
SOURCES = ["split_kernels.cu"]


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
