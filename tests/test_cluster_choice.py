"""Which form a call takes: the host code of the choice, compiled with stand-ins for the runtime's calls."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")

HEAD = """
#include <atomic>
#include <cstdio>
enum { cudaSuccess, cudaErrorUnknown };
enum { cudaFuncAttributeMaxDynamicSharedMemorySize, cudaLaunchAttributeClusterDimension };
enum { LINATTN_ERR_CUDA = -5 };
struct dim3 { unsigned x, y, z; dim3(unsigned x = 1, unsigned y = 1, unsigned z = 1) : x(x), y(y), z(z) {} };
struct cudaLaunchAttribute { int id; struct { dim3 clusterDim; } val; };
struct cudaLaunchConfig_t { dim3 gridDim, blockDim; size_t dynamicSmemBytes; cudaLaunchAttribute* attrs; int numAttrs; };
struct Problem { long long N; };
template <bool> struct Roles { static constexpr int THREADS = 1; };
template <int, bool> struct ClusterCfg { static constexpr int MOST = 8; static constexpr size_t SMEM = 1; };
template <int, bool> void umma_cluster_kernel() {}
int fail_device, fail_attribute, fail_occupancy, asked;
int cudaGetDevice(int* d) { *d = 0; return fail_device ? cudaErrorUnknown : cudaSuccess; }
int cudaGetLastError() { return 0; }
int cudaFuncSetAttribute(const void*, int, int) { return fail_attribute ? cudaErrorUnknown : cudaSuccess; }
template <class C> int cudaOccupancyMaxActiveClusters(int* n, const void*, const C* cfg) {
  static const int at_once[9] = {0, 0, 74, 45, 33, 26, 22, 15, 15};   // a B200's, one CTA to an SM
  ++asked;
  *n = at_once[cfg->attrs[0].val.clusterDim.x];
  return fail_occupancy ? cudaErrorUnknown : cudaSuccess;
}
"""


def host_code():
    text = open(os.path.join(CSRC, "umma_kernels.cu")).read()
    first = text.index("// Clusters of c CTAs that are on the device together")
    return text[first:text.index("template <int D, bool ROPE>\nint launch_cluster")]


def answers(tmp_path, main):
    src = tmp_path / "t.cpp"
    src.write_text(HEAD + host_code() + "int main() {\n" + main + "}\n")
    subprocess.run(["g++", "-std=c++17", "-o", str(tmp_path / "t"), str(src)], check=True)
    return [int(x) for x in subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout.split()]


def test_a_query_that_fails_is_an_error_and_no_other_form(tmp_path):
    """A call that the rule gives to clusters must not take the grid, with other low bits, because the runtime could not say once how
    many clusters fit."""
    out = answers(tmp_path, """
  auto size = [] { std::printf("%d\\n", cluster_size<112, true>(Problem{1200}, 4, 19, 148)); };
  fail_occupancy = 1; size(); size(); fail_occupancy = 0;
  fail_attribute = 1; size(); fail_attribute = 0;
  fail_device = 1; size(); fail_device = 0;
  size();
  int before = asked; size(); std::printf("%d\\n", asked - before);
""")
    assert out == [-5, -5, -5, -5, 8, 8, 0]


# (tokens, units) and the CTAs of a cluster: the measured points beside cluster_size
POINTS = {
    "112, true": [(128, 4, 0), (192, 4, 3), (1200, 1, 8), (6656, 1, 8), (6656, 2, 8), (6124, 4, 8), (6636, 4, 0), (5100, 6, 8), (5612, 6, 0), (4076, 8, 8),
                  (4588, 8, 0), (6636, 8, 0), (4076, 12, 8), (4588, 12, 0), (6636, 14, 8), (3052, 16, 6), (3436, 16, 0), (4588, 18, 6), (4972, 18, 0),
                  (4680, 20, 6), (4680, 22, 6), (4992, 22, 6), (4993, 22, 0), (4000, 26, 5), (3328, 33, 4), (2284, 35, 3), (2476, 35, 0), (2400, 40, 3),
                  (1004, 46, 2), (1132, 46, 0), (1516, 50, 2), (1536, 60, 2), (1537, 60, 0), (1536, 74, 2), (1200, 75, 0)],
    "112, false": [(128, 4, 0), (129, 4, 3), (1024, 4, 8), (1025, 4, 0), (600, 20, 6), (768, 20, 6), (769, 20, 0), (512, 33, 4), (513, 33, 0), (2304, 40, 3),
                   (2305, 40, 0), (1004, 46, 2), (1132, 46, 0), (1516, 50, 2), (1536, 60, 2), (192, 75, 0)],
    "64, true": [(6656, 2, 8), (6124, 8, 8), (6636, 8, 0), (6636, 12, 8), (4680, 18, 6), (1536, 46, 2)],
    "64, false": [(2048, 4, 8), (2049, 4, 0), (1024, 33, 4), (2304, 35, 3), (1388, 46, 2), (1516, 46, 0), (1536, 74, 2)],
    "32, true": [(6656, 1, 8), (6636, 5, 0), (6636, 15, 8), (4680, 22, 6)],
    "32, false": [(192, 1, 3), (2304, 45, 3), (1516, 48, 0), (1536, 60, 2)],
    "128, true": [(2048, 4, 8), (2049, 4, 0), (1536, 18, 6), (512, 74, 2)],
    "128, false": [(129, 18, 3), (192, 45, 3), (192, 46, 0), (193, 18, 0)],
}


@pytest.mark.parametrize("kernel", POINTS)
def test_the_line_lies_where_it_was_measured(tmp_path, kernel):
    calls = "".join('  std::printf("%%d\\n", cluster_size<%s>(Problem{%d}, %d, %d, 148));\n' % (kernel, N, U, -(-N // 64)) for N, U, _ in POINTS[kernel])
    assert [(N, U, c) for (N, U, _), c in zip(POINTS[kernel], answers(tmp_path, calls))] == POINTS[kernel]
