"""Which form a call takes: the host code of the choice, compiled with stand-ins for the runtime's calls."""
import os
import subprocess

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
  auto size = [] { std::printf("%d\\n", cluster_size<112, true>(Problem{1200}, 4, 19)); };
  fail_occupancy = 1; size(); size(); fail_occupancy = 0;
  fail_attribute = 1; size(); fail_attribute = 0;
  fail_device = 1; size(); fail_device = 0;
  size();
  int before = asked; size(); std::printf("%d\\n", asked - before);
""")
    assert out == [-5, -5, -5, -5, 8, 8, 0]
