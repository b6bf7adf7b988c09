"""Which grids of clusters may start early: the rule, compiled alone, and that every launch of clusters asks it."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")
AT_ONCE = {1: 148, 2: 74, 3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15, 9: 0}   # a B200's, one CTA to an SM

# (CTAs, units, tiles a CTA): the measured points beside the rule
EARLY = [(2, 74, 12), (4, 33, 12), (6, 22, 13), (8, 15, 13), (7, 15, 1), (3, 42, 12), (3, 40, 12), (3, 33, 12), (5, 24, 12), (5, 22, 12), (3, 44, 1), (3, 43, 4),
         (5, 25, 4), (1, 148, 9), (3, 80, 12)]
NOT_EARLY = [(3, 45, 1), (3, 45, 4), (3, 45, 12), (3, 44, 4), (3, 44, 12), (3, 43, 12), (5, 26, 1), (5, 26, 12), (5, 25, 12), (3, 90, 12)]


def test_the_rule(tmp_path):
    text = open(os.path.join(CSRC, "common.cuh")).read()
    rule = re.search(r"inline bool clusters_start_early\(.*?\n}\n", text, re.S).group(0)
    calls = "".join(f'  std::printf("%d\\n", (int)clusters_start_early({c}, {u}, {AT_ONCE[c]}, {AT_ONCE[c + 1]}, {n}));\n' for c, u, n in EARLY + NOT_EARLY)
    src = tmp_path / "t.cpp"
    src.write_text("#include <cstdio>\n" + rule + "int main() {\n" + calls + "}\n")
    subprocess.run(["g++", "-std=c++17", "-o", str(tmp_path / "t"), str(src)], check=True)
    out = [int(x) for x in subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout.split()]
    assert out == [1] * len(EARLY) + [0] * len(NOT_EARLY)


@pytest.mark.parametrize("file", ["umma_kernels.cu", "split_kernels.cu"])
def test_launches_of_clusters_ask(file):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    for launch in re.findall(r"at\[1\] = early_start\(\);.*?cudaLaunchKernelEx", text, re.S):   # clusters have the attribute second
        assert "cfg.numAttrs = early ? 2 : 1;" in launch
    assert text.count("at[1] = early_start();") == text.count("early = clusters_start_early(") == 1
