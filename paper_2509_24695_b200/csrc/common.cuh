// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "linattn.h"

namespace linattn {

// A descriptor with its strides resolved for one call.
struct Problem {
  int B, H, d;
  int dtype;
  long long sb, sn, sh;  // element strides of (batch, token, head); the feature axis is contiguous
  long long N;           // tokens in this call
  __host__ __device__ int units() const { return B * H; }
  __host__ __device__ long long state_elems() const { return (long long)(d + 1) * d; }  // floats per (b,h) state
};

// Control block at the start of every workspace.
struct WorkspaceCtrl {
  int status;            // LINATTN_OK or LINATTN_ERR_TIMEOUT, written by kernels
  int gave_up;           // a CTA has no partial state to give (split_state_kernel); fma_state_reduce clears it again
  int gave_up_seen;      // its blocks that have looked
  int pad0[13];
  unsigned barrier[16];  // grid-barrier counters of the fused kernels
  unsigned unit_arrivals[960];
};
static_assert(sizeof(WorkspaceCtrl) <= LINATTN_WORKSPACE_CTRL_BYTES, "control block too large");

// A kernel launched with this may be set up while the one before it in the stream is still running (programmatic dependent
// launch); nothing that it does to memory stands before its wait_for_prior_grids().  That takes the launch, and what a kernel
// does before its first load (barriers, zeros), off the time of calls in a row: back to back, forward of 192
// tokens, 4 heads of 32 12.3 -> 10.0 us, rotary read-only step of 4680 tokens 38.8 -> 35.6, temporal convolution of three 480p
// frames 14.3 -> 11.6, bf16 read-only step of 114 tokens, 56 heads of 40 (two kernels) 18.4 -> 13.1.  Cooperative kernels, which
// fill the chip, do not gain by it; fma_state_reduce neither (see there).
inline cudaLaunchAttribute early_start() {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  return at;
}
// May a grid of `units` clusters of c CTAs start early?  `at_once`, `wider`: clusters of c and of c + 1 that the device holds; share: tiles of a CTA.
//
// Not where clusters of three or five take nearly all the room that there is for them: those that are placed while the grid before is
// still leaving lie so that the last ones find no place before others are done.  (Even numbers of CTAs do not show it, and seven take
// the room of eight.)  Without early starts, with them in a row, with them behind a temporal convolution of 1560 positions; time of the read-only
// rotary step, heads of 112 (a unit each), relative to the first, by units and 64-token tiles a CTA:
//   clusters of 3 (45 at once)  45 units    1 tile .95 1.25   4 .95 1.34   12 1.26 1.49
//                               44                 .92 1.13     .90 1.18      1.09 1.34
//                               43                 .92 1.00     .90 1.02       .97 1.11
//                               42                 .92  .92     .90  .93       .92 1.00
//   clusters of 5 (26 at once)  26                 .92 1.18    1.05 1.22      1.24 1.32
//                               25                 .89  .99     .94 1.01      1.00 1.12
//                               24                 .86  .92     .93  .91       .96  .96
//   of 2, 4, 6, 8, all that fit                    .84 to .90   .89 to .93     .91 to .95
// fp32 steps of 600 and 1200 tokens (18 and 37 tiles of 32, behind the apply pass of the one before) 45 units 1.40, 44 1.35, 43 1.15, 42 1.02,
// 41 .95.  (Where the two columns disagree, few tiles a CTA, they cancel out: those start early.)
inline bool clusters_start_early(int c, long long units, int at_once, int wider, long long share) {
  if (c < 3 || c % 2 == 0 || units <= wider) return true;
  const long long spare = ((units + at_once - 1) / at_once * at_once - units) * c;   // SMs, in the last wave
  return spare > 6 || share <= spare;
}
template <typename... P, typename... A>
cudaError_t launch_early(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const A&... args) {
  cudaLaunchAttribute at[1] = {early_start()};
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#ifdef __CUDACC__
// Tensor memory is allocated between the two calls below: behind the wait, since a CTA of the grid before that is on the same SM and has
// yet to allocate its own would wait for this one, which waits for it; and before the next grid may start, for the same reason.
//
// All grids before this one in the stream are complete and what they wrote is seen.  (Loads that the compiler may take for free to
// move, __ldg, __ldcg and __ldcs, want a pointer from behind_wait; copies, bulk copies and what functions that are not inlined load stay where they are.)
__device__ __forceinline__ void wait_for_prior_grids() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename T>
__device__ __forceinline__ T* behind_wait(T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
// The next grid in the stream may be set up, as far as there is room beside this one (when every CTA has said so or left).
__device__ __forceinline__ void let_next_grid_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Kernel-launch counter behind linattn_kernel_launches().
void count_launches(int n);

constexpr int kMaxCtas = 256;        // upper bound on the persistent grid (B200 has 148 SMs)
// CTAs that ask for this much shared memory are alone on their SM (228 KB, 1 KB of it the system's per CTA).  Every kernel
// whose CTAs wait for one another (grid barriers, clusters) does: the allocation of tensor memory waits for whoever holds
// it, so CTAs of two such launches sharing two SMs could wait for each other for good.
constexpr int kSmemAlone = 114 * 1024;
static_assert(2 * (kSmemAlone + 1024) > 228 * 1024, "alone on an SM");
constexpr int kFmaMaxChunks = 64;    // split-N partials per unit on the fp32-accurate path
constexpr int kFmaMinChunkTokens = 512;

inline int fma_chunks(long long N) {
  long long p = (N + kFmaMinChunkTokens - 1) / kFmaMinChunkTokens;
  if (p < 1) p = 1;
  return p > kFmaMaxChunks ? kFmaMaxChunks : (int)p;
}

// ---- fp32-accurate path (fp32 I/O, and bf16 shapes the fused kernel does not take) ----
// state_out = (base ? base : 0) + state of tokens [0, N), base may be state_out itself; partials is scratch.
// rope: Eq. 2 with its rotary factors, table [N][d/2] of (cos, sin) fp16 pairs, one per pair rotation.
cudaError_t fma_state(const Problem& p, const void* k, const void* v, float* state_out, const float* base,
                      float* partials, WorkspaceCtrl* ctrl, cudaStream_t stream, const __half2* rope = nullptr);
cudaError_t fma_apply(const Problem& p, const void* q, const float* state, void* o, float eps, WorkspaceCtrl* ctrl, cudaStream_t stream,
                      const __half2* rope = nullptr);
// The same on the tensor cores (split_kernels.cu); ctrl: the workspace's control block.
bool split_ok(const Problem& p, const void* a, const void* b, const __half2* rope);
// *P = 0: `state` is complete ((base ? base : 0) + the tokens' state); otherwise *P partial states per unit are to be summed.
cudaError_t split_state(const Problem& p, const void* k, const void* v, const float* base, float* state, float* partials,
                        const __half2* rope, int* P, WorkspaceCtrl* ctrl, cudaStream_t stream);
cudaError_t split_apply(const Problem& p, const void* q, const float* state, void* o, float eps, const __half2* rope,
                        WorkspaceCtrl* ctrl, cudaStream_t stream);
// blk: [B][M][H][(d+1)*d] per-block states -> running states after each block (on top of cache [B][H][..]), cache := last.
cudaError_t prefix_states(float* blk, float* cache, int B, int M, long long floats_per_batch, cudaStream_t stream);
cudaError_t rope_pack(const float* cs, const float* sn, long long count, __half2* out, cudaStream_t stream);

// ---- tensor-core (tcgen05 + TMA) kernel, bf16, d in {32 (heads contiguous), 64, 112, 128} ----
// One launch runs the state pass (k, v non-null), the apply pass (q, o non-null), or both back to back.
struct UmmaCall {
  const void* k;
  const void* v;
  const void* q;
  void* o;
  float* state;     // written by the state pass, read by the apply pass
  const float* state_base;  // `accumulate`: the reduce adds the new state to this one (may be `state` itself)
  bool accumulate;
  float eps;
  const void* rope;  // rotary variant (Eq. 2 with its rotary factors): packed (cos, sin) fp16 table [N][d/2]; else null
  int blocks = 0;        // above 1: a prefill, whose batch entries are that many blocks of each entry of `cache` ...
  float* cache = nullptr;  // ... which is read and written; `state` is room for the blocks' states, and behind the partials
};
bool umma_supported(const Problem& p);
size_t umma_partial_bytes(const Problem& p, bool rope = false);
bool umma_rope_supported(const Problem& p);
// CTAs of the cluster that takes a unit of this shape (0: a lone CTA or the grid), or an error status.
int umma_cluster_ctas(const Problem& p, bool rope);
// Does a prefill of p.B / blocks entries of that many blocks of p.N tokens go in one launch (UmmaCall::blocks)?
bool umma_joins_prefill(const Problem& p, int blocks);
// Returns LINATTN_OK or an error status.
int umma_run(const Problem& p, const UmmaCall& call, void* workspace, cudaStream_t stream);

}  // namespace linattn
