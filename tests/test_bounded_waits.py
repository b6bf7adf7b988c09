"""Device-side waits give up after about a second and say so by their result.  A kernel that does not look at it goes on with
operands that never came: no call may drop the result."""
import glob
import os
import re
import subprocess

import pytest

from paper_2509_24695_b200 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")
SOURCES = sorted(os.path.basename(f) for f in build.sources() + glob.glob(os.path.join(CSRC, "*.cuh")))


def dropped(text):
    """Lines on which a call of mbar_wait or mbar_wait_cluster is a statement of its own."""
    text = re.sub(r"//[^\n]*", "", text)
    return [text.count("\n", 0, m.start()) + 1 for m in re.finditer(r"\bmbar_wait(_cluster)?\s*\(", text) if text[:m.start()].rstrip()[-1] in ";{})"]


def test_the_check_sees_a_dropped_result():
    assert len(dropped("if (t) mbar_wait(a, 0, f);")) == 1 and len(dropped("x = 1;\n  mbar_wait(a, 0, f);")) == 1
    assert not dropped("if (!mbar_wait(a, 0, f)) break; ok = mbar_wait(b, 1, f); __all_sync(m, mbar_wait(c, 1, f));")
    assert len(dropped("x = 1;\n  mbar_wait_cluster(a, 0, f);")) == 1 and not dropped("bool ok = mbar_wait_cluster(a, 0, f);")


def test_every_file_with_a_wait_is_read():
    with_waits = {os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*")) if "mbar_wait" in open(f).read()}
    assert {"umma_kernels.cu", "umma_cluster.cuh", "split_kernels.cu"} <= with_waits <= set(SOURCES)


@pytest.mark.parametrize("name", SOURCES)
def test_no_result_is_dropped(name):
    lines = dropped(open(os.path.join(CSRC, name)).read())
    assert not lines, f"{name}: a wait's result is dropped on lines {lines}"


@pytest.mark.parametrize("statement,compiles", [("if (!mbar_wait(b, 0, f)) return;", True), ("mbar_wait(b, 0, f);", False),
                                                ("if (!mbar_wait_cluster(b, 0, f)) return;", True), ("mbar_wait_cluster(b, 0, f);", False)])
def test_the_build_refuses_a_dropped_result(tmp_path, statement, compiles):
    src = tmp_path / "t.cu"
    src.write_text('#include "sm100_ptx.cuh"\n__global__ void t(uint64_t* b, volatile int* f) { using namespace linattn::ptx; %s }\n' % statement)
    rc = subprocess.run(["nvcc", *build.NVCC_FLAGS, "-I", CSRC, "-c", str(src), "-o", str(tmp_path / "t.o")], capture_output=True).returncode
    assert (rc == 0) == compiles


def struct_text(text, name):
    """The definition of `name` (with its template head, if any) in a source file."""
    m = re.search(r"(template <[^\n]*>\n)?(struct|__host__ __device__ constexpr int) %s\b[^;{]*\{" % re.escape(name), text)
    depth, end = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
    return text[m.start():end] + ";\n"


def test_ctas_that_wait_for_one_another_do_not_share_an_sm(tmp_path):
    """The CTAs of a cluster (split_state_kernel, umma_cluster_kernel) and those of a grid with barriers (umma_fused_kernel) wait for one another, and
    the allocation of tensor memory waits for whoever holds it.  Two such launches sharing two SMs could wait for each other for
    good, so each CTA has to ask for more than half of an SM's 228 KB of shared memory (1 KB of it the system's, per CTA)."""
    split = open(os.path.join(CSRC, "split_kernels.cu")).read()
    umma = open(os.path.join(CSRC, "umma_kernels.cu")).read()
    cluster = open(os.path.join(CSRC, "umma_cluster.cuh")).read()
    common = open(os.path.join(CSRC, "common.cuh")).read()
    consts = [m.group(0) for src in (common, split, umma) for m in
              re.finditer(r"^constexpr (?:int|size_t) k\w+ = [^;]*;", src, re.M) if "sizeof" not in m.group(0)]
    pieces = "".join("template <> struct Piece<%s> { static constexpr int E = %d; using Tab = Bytes<%d>; };\n" % x
                     for x in (("float", 4, 8), ("__nv_bfloat16", 8, 16)))
    asks = ["StateShape<%s, %d, %s>::SMEM" % (t, r, rope) for t in ("float", "__nv_bfloat16") for r in range(2, 9) for rope in ("false", "true")]
    asks += ["(int)Cfg<%d>::%s" % (d, s) for d in (32, 64, 112, 128) for s in ("SMEM", "SMEM_ROPE")]
    asks += ["(int)ClusterCfg<%d, %s>::SMEM" % (d, rope) for d in (32, 64, 112, 128) for rope in ("false", "true")]
    src = tmp_path / "t.cpp"
    src.write_text("#include <cstddef>\n#include <cstdint>\n#include <cstdio>\n#define __host__\n#define __device__\n"
                   "template <int N> struct Bytes { char b[N]; };\nstruct __nv_bfloat16 { char b[2]; };\ntemplate <typename T> struct Piece;\n"
                   + pieces + "\n".join(dict.fromkeys(consts)) + "\n"
                   + "".join(struct_text(split, n) for n in ("flip_of", "Shape", "StateShape")).replace("};\n;", "};\n")
                   + struct_text(umma, "Cfg") + struct_text(cluster, "ClusterCfg")
                   + "int main() {\n" + "".join('  printf("%s %%d\\n", %s);\n' % (a.replace(" ", ""), a) for a in asks) + "}\n")
    subprocess.run(["g++", "-std=c++17", "-o", str(tmp_path / "t"), str(src)], check=True)
    asked = dict(line.rsplit(" ", 1) for line in subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout.splitlines())
    assert len(asked) == len(asks)
    shared = {name: int(n) for name, n in asked.items() if 2 * (int(n) + 1024) <= 228 * 1024}
    assert not shared, f"two CTAs fit on an SM: {shared}"
