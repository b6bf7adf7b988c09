"""csrc/binding.cpp, where the interpreter's lock is let go: nothing but the library is called there.  What torch throws becomes a Python
error, which wants the lock."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc", "binding.cpp")


def test_only_the_library_is_called_without_the_lock():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    parts = re.findall(r"Py_BEGIN_ALLOW_THREADS(.*?)Py_END_ALLOW_THREADS", text, re.S)
    assert len(parts) == text.count("Py_BEGIN_ALLOW_THREADS") == 4
    for part in parts:
        calls = re.findall(r"([\w>.:-]+|\))\s*(?:<[^<>]*>)?\s*\(", part)   # what is called; ")" where a choice of two is
        called = [c for c in calls if c not in ("=", "if", "else")]
        assert called and all(re.fullmatch(r"p_\w+|\)", c) for c in called), called
