// Tensor-core kernel for bf16 ReLU linear attention on sm_100a: TMA tiles into shared memory, a ReLU
// pass in place, tcgen05.mma with fp32 accumulators in tensor memory, results streamed out.
//
// Both contractions of the method are dense and run on the tensor cores, but the work is HBM-bound
// (about d/2 FLOP per byte); everything here is organised around keeping TMA loads in flight on every SM.
//
// ONE persistent, cooperatively launched kernel runs up to three passes back to back (units of few tokens apart, see below):
//
//   state pass   S = sum_n phi(k_n)^T v_n and z = sum_n phi(k_n)   (Eq. 2 / Eq. 3 state).
//                A = phi(K)^T and B = [V | 1] are both token-major in memory, i.e. MN-major UMMA
//                operands; the contraction index is the token.  The "ones" column makes z fall out of
//                the same MMA as one more accumulator column.  Work is split over tokens across the
//                grid (split-N); every CTA writes one fp32 partial record per unit segment it covered.
//   reduce       after a grid barrier the state is summed over the partial records in a fixed order
//                (deterministic), optionally on top of the existing state: the cache update of Eq. 3.
//                Either every CTA sums a slice of the whole state, or (one-head units, fused launch) the
//                CTAs of a unit share its reduce and also leave the unit's apply operand (S as bf16
//                hi + lo, z as one more row, in the shared-memory layout) in a per-unit image.  A second
//                grid barrier publishes state and images.
//   apply pass   o_n = phi(q_n) S / (phi(q_n).z + eps).  A = phi(Q) tile (K-major), B = S split into
//                bf16 hi + lo parts (two MMAs per K step, so S keeps ~16 mantissa bits), with z as an
//                extra row of B so the denominator is one more accumulator column.  B comes into shared
//                memory once per unit segment: one bulk copy of the unit's image, or built from the fp32
//                state.  phi(Q) gets to the tensor core through tensor memory (QT below), in the lone CTAs' and the rotary
//                form through shared memory.  The epilogue divides, rounds to bf16 and a dedicated warp TMA-stores the tile.
//
// A prefill of several blocks is one launch too: its reduce also forms the running sums over the blocks (reduce_prefix).
//
// The first Q tiles of the apply pass are fetched before the grid barriers (Q does not depend on the
// state), so HBM stays busy while the partials are reduced.
//
// Head dims 32 and 64 pack four / two heads into one 128-feature operand (the cross-head blocks of the
// product are ignored / zero); 112 pads to 128 through TMA out-of-bounds zero fill.
//
// A unit of few tokens is taken by one CTA from its first token to its last output instead (SOLO): no grid barrier, no
// record, no reduce, and an ordinary launch.  Between the two, the CTAs of a unit are a cluster (umma_cluster.cuh).
//
// Warp roles (352 threads): warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2-5 ReLU
// pass, warps 6-9 epilogue, warp 10 output stores.  All cross-role synchronisation is by mbarriers
// with bounded waits, and the grid barrier is bounded too; a wait that runs out raises a CTA-wide
// abort flag, records LINATTN_ERR_TIMEOUT in the workspace status word, and every role falls through
// to the common teardown (TMEM is freed, loads in flight are waited for with a bound).
#include <cuda.h>

#include <atomic>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace linattn {
namespace {

using namespace ptx;

// Warp roles: warp 0 TMA producer, warp 1 MMA issuer, then the ReLU warps, four epilogue warps, one store
// warp.  The rotary variant does several times the arithmetic per element in the ReLU role (rotation,
// sums for z, denominators), so it runs that role on eight warps instead of four.
template <bool ROPE>
struct Roles {
  static constexpr int RELU_WARPS = ROPE ? 8 : 4;
  static constexpr int RELU_THREADS = RELU_WARPS * 32;
  static constexpr int EPI_WARP0 = 2 + RELU_WARPS;
  static constexpr int EPI_THREAD0 = EPI_WARP0 * 32;
  static constexpr int STORE_WARP = EPI_WARP0 + 4;
  static constexpr int THREADS = (STORE_WARP + 1) * 32;
};
constexpr int kReluThread0 = 64;
constexpr int kTileApply = 128;     // tokens per apply tile (= UMMA M)
constexpr int kTileState = 64;      // tokens per state stage (4 UMMA K steps of 16 tokens)
constexpr int kRowBytes = 128;      // one swizzle row: 64 bf16
constexpr int kBox = kTileState * kRowBytes;  // 8 KB: one 64-feature box of a state stage
constexpr int kTmemCols = 512;
constexpr int kAccStride = 256;     // TMEM columns between the two accumulator buffers

// rotary variant: floats a partial record carries for z: per warp that sums plain phi(k) (the eight ReLU warps, and
// the four epilogue warps, which take a share of the second K box in the state pass), per feature
constexpr int kZSlots = 12;
constexpr int kZParts = kZSlots * 128;

template <int D>
struct Cfg {
  static constexpr int G = D == 32 ? 4 : D == 64 ? 2 : 1;   // heads packed into one 128-feature operand
  static constexpr int FEAT = G * D;                         // 112 or 128 live features per group
  static constexpr int KSTEPS = FEAT / 16;                   // apply: K steps over features
  static constexpr int ZROW = D == 112 ? 112 : 128;          // apply: accumulator column of the first denominator
  static constexpr int NAPPLY = D == 112 ? 128 : 144;        // apply MMA N
  // state: with D = 112 the 1 sits in value column 112 (zero padding the TMA wrote), else in a
  // constant extra chunk of the stage
  static constexpr bool ONES_BOX = D != 112;
  static constexpr int NSTATE = ONES_BOX ? 144 : 128;        // state MMA N
  static constexpr int ZCOL = ONES_BOX ? 128 : 112;          // state accumulator column that holds z
  // The tensor core truncates when it adds into the fp32 accumulator, so a long chain of updates drifts
  // (about 2^-24 relative per update).  The state pass therefore deals its MMAs round-robin to several
  // accumulators, which the epilogue adds up (round to nearest) once per segment: shorter chains.
  static constexpr int STATE_ACCS = ONES_BOX ? 3 : 4;
  static constexpr int STATE_ACC_STRIDE = ONES_BOX ? 160 : 128;   // TMEM columns between them
  static constexpr int BOX_D = 64;                           // TMA box: features ...
  static constexpr int BOX_H = 1;                            // ... x heads
  static constexpr int SBOX_BYTES = NAPPLY * kRowBytes;      // one 64-feature K box of the S operand
  static constexpr int S_BYTES = 4 * SBOX_BYTES;             // (hi, lo) x 2 K boxes
  static constexpr int APPLY_SLOTS = D == 112 ? 5 : 4;
  static constexpr int SLOT_BYTES = 2 * kTileApply * kRowBytes;        // 32 KB: two 64-feature boxes
  static constexpr int STAGE_BYTES = (ONES_BOX ? 5 : 4) * kBox;        // V0 V1 [ONES] K0 K1
  static constexpr int KOFF = (ONES_BOX ? 3 : 2) * kBox;               // K boxes within a stage
  static constexpr int DATA_BYTES = S_BYTES + APPLY_SLOTS * SLOT_BYTES;
  // The data area would hold up to seven stages, but four measured fastest: with more bytes in flight
  // per SM the memory system's queues grow and the SMs' shares of the bandwidth drift apart.
  static constexpr int STATE_STAGES = DATA_BYTES / STAGE_BYTES < 4 ? DATA_BYTES / STAGE_BYTES : 4;
  static constexpr int BAR_BYTES = 1024;
  // rotary variant without row padding (every head dim but 112): the denominators of a tile's rows travel in a small
  // array per slot and head of the group
  static constexpr int DEN_BYTES = D == 112 ? 0 : G * APPLY_SLOTS * kTileApply * 4;
  static constexpr size_t SMEM = 1024 + DATA_BYTES + BAR_BYTES;
  static constexpr size_t SMEM_ROPE = SMEM + DEN_BYTES;
  // Rotary variant, state pass of the grid form: the stage holds the rotations of its 64 tokens behind V0 V1 K0 K1.
  static constexpr int TAB_ROW = 2 * D;                      // d/2 (cos, sin) fp16 pairs
  static constexpr int ROPE_STAGE_BYTES = 4 * kBox + kTileState * TAB_ROW;
  static constexpr int ROPE_STAGES = 4;
  static_assert(ROPE_STAGES * ROPE_STAGE_BYTES <= DATA_BYTES, "stages of the rotary variant");
  // lone CTAs (see solo_drain): the slots, then the warps' sums for z and z, then the unit's state as it is in memory
  static constexpr int SOLO_SLOTS = D == 128 ? 2 : 3;
  static constexpr int SOLO_STAGE_BYTES = 4 * kBox;            // no "ones"
  static constexpr int SOLO_Z = S_BYTES + SOLO_SLOTS * SLOT_BYTES, SOLO_STATE = SOLO_Z + (kZSlots + 1) * 128 * 4;
  static constexpr int SOLO_DATA = (SOLO_STATE + G * (D + 1) * D * 4 + 127) & ~127;
  static constexpr size_t SMEM_SOLO = 1024 + SOLO_DATA + BAR_BYTES + DEN_BYTES;
  static_assert(4 * SOLO_STAGE_BYTES <= SOLO_Z && SMEM_SOLO <= 227 * 1024, "shared memory of a lone CTA");
  // rotary variant: 16-byte chunk of a token's table row (d/2 fp16 pairs) that goes with logical chunk lc of box 0 / 1.
  // With packed heads (d = 32, 64) box 1 starts a new head, so both boxes use the same chunk.
  static constexpr bool SAME_TAB = 64 % D == 0;
  __host__ __device__ static constexpr int tab_chunk(int box, int lc) { return ((64 * box + 8 * lc) % D) / 8; }
};

// How the (unit, token tile) work of one pass is dealt to the persistent grid.
//
// A unit is one (batch, head group); its tiles are consecutive token ranges.  With U units and `grid`
// CTAs, the first P*U CTAs ("column" CTAs, P = grid / U) take tiles [c*Lc, (c+1)*Lc) of unit j % U with
// c = j / U and Lc = ceil(U*tpu / grid); the remaining R CTAs split the tiles [P*Lc, tpu) of all units
// evenly, unit after unit.  Column CTAs of neighbouring heads therefore walk the same token range at
// the same time.  That matters for head dims whose rows are not whole 128-byte lines (112 features =
// 224 bytes): a line shared by two heads comes from DRAM once if both heads ask for it while it is
// still in L2, and twice if their CTAs reach it tens of microseconds apart.
struct Sched {
  int U, tpu, grid;
  int P, Lc, R;
  int m;  // tiles per unit left to the R trailing CTAs: tpu - min(P*Lc, tpu)
};

// One CTA's share: flat positions [f0, f1); position f is tile tile_base + f % mm of unit
// unit_base + f / mm, and the partial record of that unit's segment is rec_base + f / mm.
struct Work {
  long long f0, f1;
  int mm, tile_base, unit_base, rec_base;
};

__host__ __device__ inline Work work_of(const Sched& s, int j) {
  Work w;
  w.f0 = w.f1 = 0; w.mm = 1; w.tile_base = 0; w.unit_base = 0; w.rec_base = 0;
  if (j >= s.grid) return w;
  if (j < s.P * s.U) {
    const int t0 = (j / s.U) * s.Lc;
    const int t1 = t0 + s.Lc < s.tpu ? t0 + s.Lc : s.tpu;
    w.f1 = t1 > t0 ? t1 - t0 : 0;
    w.mm = 0x7fffffff; w.tile_base = t0; w.unit_base = j % s.U; w.rec_base = j;
  } else {
    const int r = j - s.P * s.U;
    const long long tot = (long long)s.U * s.m;
    w.f0 = r * tot / s.R; w.f1 = (r + 1) * tot / s.R;
    w.mm = s.m > 0 ? s.m : 1; w.tile_base = s.P * s.Lc; w.rec_base = s.P * s.U + r;
  }
  return w;
}

// `seg_cost`: what starting one more unit segment costs a CTA, in tiles (drain of the accumulators /
// rebuild of the S operand).  Trailing CTAs cross several units, so the columns are made a little longer
// until the trailing CTAs' tiles plus their segment starts fit into a column's time.
inline Sched make_sched(int U, long long tpu, int max_ctas, int seg_cost) {
  Sched s;
  const long long total = (long long)U * tpu;
  s.U = U; s.tpu = (int)tpu;
  s.grid = (int)(total < max_ctas ? total : max_ctas);
  if (s.grid < 1) s.grid = 1;
  s.P = s.grid / U;
  s.R = s.grid - s.P * U;
  const int lc0 = (int)((total + s.grid - 1) / s.grid);
  s.Lc = lc0;
  if (s.P > 0 && s.R > 0) {
    for (int lc = lc0; lc < lc0 + 8; ++lc) {
      const long long m = (long long)s.P * lc >= tpu ? 0 : tpu - (long long)s.P * lc;
      const long long tiles = (U * m + s.R - 1) / s.R;
      const long long segs = m > 0 ? (tiles + m - 1) / m + 1 : 0;
      if (tiles + segs * seg_cost <= lc) { s.Lc = lc; break; }
    }
  }
  const long long covered = (long long)s.P * s.Lc;
  s.m = covered >= tpu ? 0 : (int)(tpu - covered);
  return s;
}

// Walks a Work range tile by tile.
struct TileWalk {
  const Work w;
  long long f;
  int uo, tp;
  __device__ explicit TileWalk(const Work& w_) : w(w_), f(w_.f0), uo((int)(w_.f0 / w_.mm)), tp((int)(w_.f0 % w_.mm)) {}
  __device__ bool done() const { return f >= w.f1; }
  __device__ int unit() const { return w.unit_base + uo; }
  __device__ int tile() const { return w.tile_base + tp; }
  __device__ int record() const { return w.rec_base + uo; }
  __device__ bool seg_first() const { return f == w.f0 || tp == 0; }
  __device__ bool seg_last() const { return f + 1 == w.f1 || tp == w.mm - 1; }
  __device__ void next() { ++f; if (++tp == w.mm) { tp = 0; ++uo; } }
};

struct FusedParams {
  int B, H, HG;            // HG: head groups per batch entry = ceil(H / G)
  Sched sa, sc;            // state pass (64-token stages) and apply pass (128-token tiles)
  int do_state, do_apply;
  int accumulate;          // reduce on top of state_base
  float* state;            // [B][H][(d+1)][d]: written by the reduce, read by the apply pass
  const float* state_base; // the state the new one is added to (the cache; may be `state` itself)
  float* partials;         // one record of G head-states per (CTA, unit) segment of the state pass
  float eps;
  WorkspaceCtrl* ctrl;
  uint8_t* s_image;        // non-null: the reduce also leaves every unit's S operand (bf16 hi + lo, in the shared-memory
                           // layout) here, S_BYTES per unit, and the apply pass fetches it with one bulk copy
  int blocks;              // prefill: batch entry b of K, V, Q, O is block b % blocks of entry b / blocks of the cache
  float* cache;            // ... [B / blocks][H][(d+1)][d]: the state before the first block, and (written) after the last one
  int write_state;         // lone CTAs: the new state goes to `state` (a launch whose state nobody reads keeps it on chip)
  const uint4* rope;       // rotary variant: [N][d/8] chunks of four (cos, sin) fp16 pairs; null otherwise
  long long N;             // tokens (bound of the rotary table)
};

// TMA coordinates (feature, head) of 64-element box `box` (0/1) of head group hg
template <int D>
__device__ __forceinline__ void box_coords(int box, int hg, int& c0, int& c1) {
  if (Cfg<D>::G == 1) { c0 = 64 * box; c1 = hg; }
  else if (Cfg<D>::G == 2) { c0 = 0; c1 = 2 * hg + box; }
  else { c0 = 128 * hg + 64 * box; c1 = 0; }  // d = 32: the map sees a token's heads as one row of H*32 features
}

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

// In-place ReLU over the two 64-feature boxes (ROWS token rows of 128 bytes each, 128-byte swizzle) of a
// tile, 128 threads, thread `t`.  A thread owns one 16-byte column position of rows t/8 + 16*i; with the
// 128-byte swizzle the logical chunk at that position is the same for all of its rows, so with FEAT = 112
// a thread whose chunk of the second box holds only zero padding (features 112..127) skips that box.
// All loads of a box are issued before the first store.
template <int FEAT, int ROWS>
__device__ __forceinline__ void relu_pass(uint8_t* box0, uint8_t* box1, int t) {
  const int row0 = t >> 3, pc = t & 7;
  const int lc = pc ^ (row0 & 7);
  uint8_t* p0 = box0 + row0 * kRowBytes + pc * 16;
  uint8_t* p1 = box1 + row0 * kRowBytes + pc * 16;
  uint4 x[ROWS / 16];
#pragma unroll
  for (int i = 0; i < ROWS / 16; ++i) x[i] = *reinterpret_cast<uint4*>(p0 + i * 16 * kRowBytes);
#pragma unroll
  for (int i = 0; i < ROWS / 16; ++i) {
    x[i].x = relu_bf16x2(x[i].x); x[i].y = relu_bf16x2(x[i].y); x[i].z = relu_bf16x2(x[i].z); x[i].w = relu_bf16x2(x[i].w);
    *reinterpret_cast<uint4*>(p0 + i * 16 * kRowBytes) = x[i];
  }
  if (FEAT >= 128 || 64 + lc * 8 < FEAT) {
#pragma unroll
    for (int i = 0; i < ROWS / 16; ++i) x[i] = *reinterpret_cast<uint4*>(p1 + i * 16 * kRowBytes);
#pragma unroll
    for (int i = 0; i < ROWS / 16; ++i) {
      x[i].x = relu_bf16x2(x[i].x); x[i].y = relu_bf16x2(x[i].y); x[i].z = relu_bf16x2(x[i].z); x[i].w = relu_bf16x2(x[i].w);
      *reinterpret_cast<uint4*>(p1 + i * 16 * kRowBytes) = x[i];
    }
  }
}

// ReLU of row r of a Q tile on its way to tensor memory: the row's features from the slot to the columns from `at` on (of this lane; a
// warp's rows are its lane quarter), two to a column, as the MMA wants its A operand there.
template <int FEAT>
__device__ __forceinline__ void relu_row_to_tmem(const uint8_t* slot, int half, int r, uint32_t at) {
  const uint8_t* row = slot + r * kRowBytes;
#pragma unroll
  for (int box = 0; box < 2; ++box) {
    uint32_t w[32];
#pragma unroll
    for (int c = 0; c < 8; ++c) {   // neighbouring rows have a chunk at different places (swizzle): no bank conflicts
      if (64 * box + 8 * c >= FEAT) break;
      const uint4 x = *reinterpret_cast<const uint4*>(row + box * half + ((c ^ (r & 7)) << 4));
      w[4 * c] = relu_bf16x2(x.x); w[4 * c + 1] = relu_bf16x2(x.y); w[4 * c + 2] = relu_bf16x2(x.z); w[4 * c + 3] = relu_bf16x2(x.w);
    }
    if (box == 0 || FEAT == 128) {
      tmem_st_x32(at + 32 * box, w);
    } else {
      static_assert(FEAT == 112 || FEAT == 128, "columns of the second box");
      tmem_st_x16(at + 32, w);
      tmem_st_x8(at + 48, w + 16);
    }
  }
  tmem_st_wait();
}

// The same, adding the plain values up per thread: z[0..3] for its chunk of box 0, z[4..7] for that of box 1.
__device__ __forceinline__ void unpack_relu8(const uint4& x, float2 (&f)[4]);
template <int FEAT, int ROWS>
__device__ __forceinline__ void relu_sum_pass(uint8_t* box0, uint8_t* box1, int t, float2 (&z)[8]) {
  relu_pass<FEAT, ROWS>(box0, box1, t);
  const int row0 = t >> 3, pc = t & 7;
  const int lc = pc ^ (row0 & 7);
#pragma unroll
  for (int box = 0; box < 2; ++box) {
    if (box == 1 && FEAT < 128 && 64 + lc * 8 >= FEAT) break;
    const uint8_t* p = (box ? box1 : box0) + row0 * kRowBytes + pc * 16;
#pragma unroll
    for (int i = 0; i < ROWS / 16; ++i) {
      float2 f[4];
      unpack_relu8(*reinterpret_cast<const uint4*>(p + i * 16 * kRowBytes), f);
#pragma unroll
      for (int e = 0; e < 4; ++e) z[4 * box + e] = add2(z[4 * box + e], f[e]);
    }
  }
}

// Rotary variant: a 16-byte chunk holds four feature pairs; `tab` holds their (cos, sin) as fp16 pairs.
// (a, b) -> (a c - b s, a s + b c), rounded to bf16.
// The clamp is done on the packed bf16 pairs, and the sums and the denominators use the packed f32x2 instructions.
__device__ __forceinline__ void unpack_relu8(const uint4& x, float2 (&f)[4]) {
  const uint32_t w[4] = {relu_bf16x2(x.x), relu_bf16x2(x.y), relu_bf16x2(x.z), relu_bf16x2(x.w)};
#pragma unroll
  for (int e = 0; e < 4; ++e) f[e] = make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xFFFF0000u));
}
__device__ __forceinline__ uint4 rotate_pack8(const float2 (&f)[4], const uint4& tab) {
  const uint32_t t[4] = {tab.x, tab.y, tab.z, tab.w};
  uint32_t o[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 cs = __half22float2(*reinterpret_cast<const __half2*>(&t[e]));
    // (scalar: the packed f32x2 forms want the cosine and the sine twice in neighbouring registers, and the pair swapped)
    o[e] = pack_bf16x2(fmaf(-f[e].y, cs.y, f[e].x * cs.x), fmaf(f[e].x, cs.y, f[e].y * cs.x));
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
constexpr uint32_t kRopeIdentity = 0x00003C00u;  // (cos, sin) = (1, 0) as an fp16 pair

// ---------------------------------------------------------------- grid barrier
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All CTAs of the (cooperatively launched, hence co-resident) grid meet here.  One word holds an arrival count
// (low 16 bits) and a generation (high 16 bits).  Before a barrier the count is pre-set to 2^16 - grid (CTA 0 adds
// that: at kernel start for the first barrier, on leaving a barrier for the next one), so the last arrival's own
// atomic add carries into the generation: the CTAs polling the word see the barrier open one L2 round trip after
// the last arrival, with no second, dependent atomic in between (that cost 0.6 us per barrier).  All updates are
// atomic adds, which commute, so the carry happens at the (grid + 1)-th add whatever their order, and the count is
// back at zero after the launch's last barrier.  Every CTA has read the generation at kernel start (it cannot
// change before the CTA's own arrival), so it knows which value to wait for and starts polling without waiting for
// the answer to its own add (0.3-0.5 us per launch); the answer is only used afterwards, as a check.  The poll is
// bounded (about a second); on expiry the CTA raises its abort flag and goes on to the teardown.
__device__ __forceinline__ void grid_barrier_preset(WorkspaceCtrl* ctrl) {
  atomicAdd(&ctrl->barrier[0], 0x10000u - gridDim.x);
}

__device__ __forceinline__ void grid_barrier(WorkspaceCtrl* ctrl, volatile int* abort_flag, bool another_follows, unsigned gen_before) {
  tcgen05_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned* word = &ctrl->barrier[0];
    // release: the CTA's writes (seen by this thread through the bar.sync) are visible before the arrival is.
    // The value the add returns is looked at only after the poll, so the poll does not wait for it.
    unsigned old;
    asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(word) : "memory");
    const unsigned long long t0 = global_timer_ns();
    while (((ld_acquire_gpu(word) >> 16) & 0xFFFFu) == (gen_before & 0xFFFFu)) {
      if (global_timer_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; break; }
    }
    // a word that was not in the state a finished launch leaves it in (count zero) can carry early: the generation
    // this CTA met at its arrival then differs from the one it read at kernel start, and the launch is given up
    if (((old >> 16) & 0xFFFFu) != (gen_before & 0xFFFFu)) *abort_flag = 1;
    if (another_follows && blockIdx.x == 0 && !*abort_flag) grid_barrier_preset(ctrl);
  }
  __syncthreads();
  tcgen05_fence_after();
}

// ---------------------------------------------------------------- reduce
// This CTA's slice of the state: state[b][h][e] = (accumulate ? state : 0) + the partial records of
// the head's unit, column CTAs first (ascending), then the trailing CTAs (ascending).
//
// The reduce sits between two grid barriers with HBM idle, so it is written for latency: a thread takes
// up to NE elements (float4) of the slice, works out where all their records are, issues every load
// (NE x NR independent 16-byte loads, plus the old state when accumulating) and only then adds, in the
// fixed order.  Index arithmetic is 32-bit wherever the sizes allow: 64-bit division is a long
// subroutine, and a handful of them per element used to cost more time than the loads.

// Trailing CTA r covers the flat positions [r*tot/R, (r+1)*tot/R) (work_of); the one that holds position f is
// the largest r with r*tot/R <= f, i.e. floor(((f+1)*R - 1) / tot): one division.
__device__ __forceinline__ int trailing_cta_of(long long f, long long tot, int R) {
  if ((tot + 1) * R < 0xffffffffLL) return (int)((((unsigned)f + 1u) * (unsigned)R - 1u) / (unsigned)tot);
  return (int)(((f + 1) * R - 1) / tot);
}

__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }

template <int D, bool ROPE, int NE, int NR>
__device__ __forceinline__ void reduce_elements(const FusedParams& p, int first, int i1, int ncol) {
  using C = Cfg<D>;
  constexpr int E4 = (D + 1) * D / 4;  // float4 per head state
  constexpr int REC4 = C::G * E4 + (ROPE ? kZParts / 4 : 0);  // float4 per partial record
  const Sched& s = p.sa;
  const long long ttot = (long long)s.U * s.m;
  float4* state4 = reinterpret_cast<float4*>(p.state);
  const float4* src[NE];
  int u_of[NE], r_lo[NE], nrec[NE];
  bool live[NE];
  float4 sum[NE], v[NE][NR];
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    const int idx = first + k * (int)blockDim.x;
    live[k] = idx < i1 && !(ROPE && idx % E4 >= D * D / 4);   // (rotary variant: z is reduce_z's)
    if (!live[k]) continue;
    sum[k] = p.accumulate ? __ldcg(reinterpret_cast<const float4*>(p.state_base) + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
    const int bh = idx / E4, e = idx - bh * E4;
    const int b = bh / p.H, h = bh - b * p.H;
    const int u = b * p.HG + h / C::G, g = h % C::G;
    u_of[k] = u;
    src[k] = reinterpret_cast<const float4*>(p.partials) + (size_t)g * E4 + e;
    int ntrail = 0;
    r_lo[k] = 0;
    if (s.m > 0) {
      r_lo[k] = trailing_cta_of((long long)u * s.m, ttot, s.R);
      ntrail = trailing_cta_of((long long)(u + 1) * s.m - 1, ttot, s.R) - r_lo[k] + 1;
    }
    nrec[k] = ncol + ntrail;
  }
  auto record_of = [&](int k, int kk) { return kk < ncol ? kk * s.U + u_of[k] : s.P * s.U + r_lo[k] + (kk - ncol) + u_of[k]; };
  int nmax = 0;
#pragma unroll
  for (int k = 0; k < NE; ++k)
    if (live[k] && nrec[k] > nmax) nmax = nrec[k];
  for (int k0 = 0; k0 < nmax; k0 += NR) {
#pragma unroll
    for (int k = 0; k < NE; ++k)
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (live[k] && k0 + r < nrec[k]) v[k][r] = __ldcg(src[k] + (size_t)record_of(k, k0 + r) * REC4);
#pragma unroll
    for (int k = 0; k < NE; ++k)
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (live[k] && k0 + r < nrec[k]) add4(sum[k], v[k][r]);
  }
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    if (!live[k]) continue;
    const int idx = first + k * (int)blockDim.x;
    state4[idx] = sum[k];
  }
}

// Rotary variant: z of all units, split evenly over the CTAs, from the plain phi(k) sums that the warps of every segment
// left behind the record.  Sixteen threads to a float4 of a unit's 128 features, one warp slot each: all of a slot's
// records in flight together, added in their fixed order; the slots are then added as a balanced tree, the missing ones
// zero (reduce_image_zrow's association).  One slot after the other in one thread, as before, this was 25 us of the 66 us
// of a rotary step of 4680 tokens, 35 heads of 64.
template <int D>
__device__ __forceinline__ void reduce_z(const FusedParams& p, int ncol) {
  using C = Cfg<D>;
  constexpr int E4 = (D + 1) * D / 4, REC4 = C::G * E4 + kZParts / 4, Z4 = C::FEAT / 4, NR = 6;
  const Sched& s = p.sa;
  const long long ttot = (long long)s.U * s.m;
  const int tot = s.U * Z4, me = (int)blockIdx.x;
  const int i0 = (int)((long long)tot * me / gridDim.x), i1 = (int)((long long)tot * (me + 1) / gridDim.x);
  const int w = (int)threadIdx.x & 15;
  for (int first = i0; first < i1; first += (int)blockDim.x / 16) {   // whole warps: the shuffles below stay inside one
    const int idx = first + (int)threadIdx.x / 16;
    const int u = idx / Z4, ft4 = idx - u * Z4;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (idx < i1 && (w < 8 || (w < kZSlots && ft4 >= 16))) {   // (features 64..: the epilogue warps' slots hold a share too)
      int r_lo = 0, nrec = ncol;
      if (s.m > 0) {
        r_lo = trailing_cta_of((long long)u * s.m, ttot, s.R);
        nrec += trailing_cta_of((long long)(u + 1) * s.m - 1, ttot, s.R) - r_lo + 1;
      }
      const float4* zp = reinterpret_cast<const float4*>(p.partials) + C::G * E4 + w * 32 + ft4;
      for (int k0 = 0; k0 < nrec; k0 += NR) {
        float4 v[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const int kk = k0 + r;
          if (kk < nrec) v[r] = __ldcg(zp + (size_t)(kk < ncol ? kk * s.U + u : s.P * s.U + r_lo + (kk - ncol) + u) * REC4);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (k0 + r < nrec) add4(acc, v[r]);
      }
    }
#pragma unroll
    for (int st = 1; st < 16; st *= 2) {
      float4 o;
      o.x = __shfl_xor_sync(0xffffffffu, acc.x, st); o.y = __shfl_xor_sync(0xffffffffu, acc.y, st);
      o.z = __shfl_xor_sync(0xffffffffu, acc.z, st); o.w = __shfl_xor_sync(0xffffffffu, acc.w, st);
      add4(acc, o);
    }
    const int g = ft4 * 4 / D, h = (u % p.HG) * C::G + g;
    if (idx < i1 && w == 0 && h < p.H) {
      const size_t e4 = ((size_t)((u / p.HG) * p.H + h) * (D + 1) + D) * (D / 4) + (ft4 - g * (D / 4));
      float4 sum = p.accumulate ? __ldcg(reinterpret_cast<const float4*>(p.state_base) + e4) : make_float4(0.f, 0.f, 0.f, 0.f);
      add4(sum, acc);
      reinterpret_cast<float4*>(p.state)[e4] = sum;
    }
  }
}

template <int D, bool ROPE>
__device__ void reduce_slice(const FusedParams& p) {
  constexpr int E4 = (D + 1) * D / 4;
  const Sched& s = p.sa;
  const int tot = p.B * p.H * E4;   // < 2^31: at most 65535 units of at most 4128 float4
  const int per = tot / (int)gridDim.x, rem = tot - per * (int)gridDim.x, me = (int)blockIdx.x;
  const int i0 = me * per + (me < rem ? me : rem);
  const int i1 = i0 + per + (me < rem ? 1 : 0);
  const int ncol = s.P == 0 ? 0 : (s.P < (s.tpu + s.Lc - 1) / s.Lc ? s.P : (s.tpu + s.Lc - 1) / s.Lc);
  if (ROPE) reduce_z<D>(p, ncol);
  // few elements per thread: more records per batch; more elements: fewer records each (about 20 loads either way;
  // half as many in the rotary variant, whose 480 threads have 128 registers each)
  if (i1 - i0 <= 2 * (int)blockDim.x) {
    for (int first = i0 + (int)threadIdx.x; first < i1; first += 2 * (int)blockDim.x)
      reduce_elements<D, ROPE, 2, ROPE ? 5 : 10>(p, first, i1, ncol);
  } else {
    for (int first = i0 + (int)threadIdx.x; first < i1; first += 3 * (int)blockDim.x)
      reduce_elements<D, ROPE, 3, ROPE ? 3 : 6>(p, first, i1, ncol);
  }
}

// ---------------------------------------------------------------- reduce, with the S operand as a by-product
// Fused launches of one-head units (d = 112, 128) with at least one column CTA per unit: the column CTAs of a
// unit share its reduce (part c of P), in 32-byte chunks of a state row, and besides the fp32 state each chunk's
// sum is split into bf16 hi + lo and stored where the apply MMA wants it (the layout build_s_operand writes to
// shared memory), in a per-unit image in the workspace.  After the second barrier a CTA gets its unit's operand
// with one bulk copy instead of re-reading and converting the whole state: the conversion is done once per
// unit, not once per CTA, and the serial section between the passes is about 2 us shorter.  Same records in the
// same order as reduce_slice, so the state comes out bit for bit the same.
template <int D, bool ROPE, int NE, int NR>
__device__ __forceinline__ void reduce_image_chunks(const FusedParams& p, int u, int first, int hi_end, int ncol, int r_lo,
                                                    int nrec) {
  using C = Cfg<D>;
  constexpr int CPR = D / 8;                 // 32-byte chunks per state row
  constexpr int E4 = (D + 1) * D / 4;        // float4 per head state
  constexpr int REC4 = E4 + (ROPE ? kZParts / 4 : 0);
  const Sched& s = p.sa;
  auto record_of = [&](int kk) { return kk < ncol ? kk * s.U + u : s.P * s.U + r_lo + (kk - ncol) + u; };
  const float4* part4 = reinterpret_cast<const float4*>(p.partials);
  float4 sum[NE][2], v[NE][NR][2];
  int j_of[NE], c_of[NE];
  bool live[NE], zrow[NE];
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    const int idx = first + k * (int)blockDim.x;
    live[k] = idx < hi_end;
    zrow[k] = false;
    if (!live[k]) continue;
    j_of[k] = idx / CPR;
    c_of[k] = idx - j_of[k] * CPR;
    zrow[k] = false;   // (rotary variant: the z row is not among the chunks, see reduce_image_zrow)
    const size_t e4 = (size_t)u * E4 + (size_t)j_of[k] * (D / 4) + 2 * c_of[k];
    if (p.accumulate) {
      sum[k][0] = __ldcg(reinterpret_cast<const float4*>(p.state_base) + e4);
      sum[k][1] = __ldcg(reinterpret_cast<const float4*>(p.state_base) + e4 + 1);
    } else {
      sum[k][0] = sum[k][1] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  for (int k0 = 0; k0 < nrec; k0 += NR) {
#pragma unroll
    for (int k = 0; k < NE; ++k)
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (live[k] && !zrow[k] && k0 + r < nrec) {
          const float4* src = part4 + (size_t)record_of(k0 + r) * REC4 + j_of[k] * (D / 4) + 2 * c_of[k];
          v[k][r][0] = __ldcg(src);
          v[k][r][1] = __ldcg(src + 1);
        }
#pragma unroll
    for (int k = 0; k < NE; ++k)
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (live[k] && !zrow[k] && k0 + r < nrec) { add4(sum[k][0], v[k][r][0]); add4(sum[k][1], v[k][r][1]); }
  }
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    if (!live[k]) continue;
    const int j = j_of[k], c = c_of[k];
    float4* dst = reinterpret_cast<float4*>(p.state) + (size_t)u * E4 + (size_t)j * (D / 4) + 2 * c;
    dst[0] = sum[k][0];
    dst[1] = sum[k][1];
    const float x[8] = {sum[k][0].x, sum[k][0].y, sum[k][0].z, sum[k][0].w, sum[k][1].x, sum[k][1].y, sum[k][1].z, sum[k][1].w};
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const __nv_bfloat16 h0 = __float2bfloat16_rn(x[2 * e]), h1 = __float2bfloat16_rn(x[2 * e + 1]);
      hi[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
      lo[e] = pack_bf16x2(x[2 * e] - __bfloat162float(h0), x[2 * e + 1] - __bfloat162float(h1));
    }
    const int jrow = j < D ? j : C::ZROW;   // operand row: value feature, or the z row
    const int i0 = c * 8;                   // first key feature of this chunk
    const int off = (i0 >> 6) * C::SBOX_BYTES + jrow * kRowBytes + ((((i0 & 63) >> 3) ^ (jrow & 7)) << 4);
    uint8_t* img = p.s_image + (size_t)u * C::S_BYTES;
    *reinterpret_cast<uint4*>(img + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(img + 2 * C::SBOX_BYTES + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// Rotary variant: z of unit u from the plain phi(k) sums that the warps of every segment left behind the record,
// [12 warp slots][128 features] (the epilogue warps' slots 8..11 only for features 64..).  Thread (float4 hc of z,
// slot w of 16) adds its slot over the records in their fixed order (all loads in flight together; slots that
// do not exist count as zero), shuffles add the sixteen as a balanced tree, lane w = 0 adds the old z when
// accumulating; two neighbouring float4 make the 32-byte chunk of the operand image.
template <int D>
__device__ __forceinline__ void reduce_image_zrow(const FusedParams& p, int u, int ncol, int r_lo, int nrec) {
  using C = Cfg<D>;
  constexpr int E4 = (D + 1) * D / 4, REC4 = E4 + kZParts / 4, Z4 = D / 4, NR = 6;
  static_assert((16 * Z4) % 32 == 0 && Z4 % 2 == 0, "whole warps take part in the shuffles");
  // sixteen threads per float4 of z; with fewer than 16 * Z4 threads (d = 128: 512 wanted, 480 there) the first warps
  // take a second turn (whole warps: the shuffles below stay inside a warp)
  for (int t = (int)threadIdx.x; t < 16 * Z4; t += ((int)blockDim.x / 32) * 32) {
  const int hc = t >> 4, w = t & 15;
  const Sched& s = p.sa;
  auto record_of = [&](int kk) { return kk < ncol ? kk * s.U + u : s.P * s.U + r_lo + (kk - ncol) + u; };
  const float4* zp = reinterpret_cast<const float4*>(p.partials) + E4 + w * 32 + hc;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (w < 8 || (w < kZSlots && hc >= 16)) {
    for (int k0 = 0; k0 < nrec; k0 += NR) {
      float4 v[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (k0 + r < nrec) v[r] = __ldcg(zp + (size_t)record_of(k0 + r) * REC4);
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (k0 + r < nrec) add4(acc, v[r]);
    }
  }
#pragma unroll
  for (int st = 1; st < 16; st *= 2) {
    float4 o;
    o.x = __shfl_xor_sync(0xffffffffu, acc.x, st); o.y = __shfl_xor_sync(0xffffffffu, acc.y, st);
    o.z = __shfl_xor_sync(0xffffffffu, acc.z, st); o.w = __shfl_xor_sync(0xffffffffu, acc.w, st);
    add4(acc, o);
  }
  const size_t e4 = (size_t)u * E4 + (size_t)D * (D / 4) + hc;
  float4 sum = p.accumulate ? __ldcg(reinterpret_cast<const float4*>(p.state_base) + e4) : make_float4(0.f, 0.f, 0.f, 0.f);
  add4(sum, acc);
  float4 up;   // the upper half of this chunk, from the lane that holds float4 hc + 1
  up.x = __shfl_xor_sync(0xffffffffu, sum.x, 16); up.y = __shfl_xor_sync(0xffffffffu, sum.y, 16);
  up.z = __shfl_xor_sync(0xffffffffu, sum.z, 16); up.w = __shfl_xor_sync(0xffffffffu, sum.w, 16);
  if (w != 0) continue;
  reinterpret_cast<float4*>(p.state)[e4] = sum;
  if (hc & 1) continue;
  const float x[8] = {sum.x, sum.y, sum.z, sum.w, up.x, up.y, up.z, up.w};
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat16 h0 = __float2bfloat16_rn(x[2 * e]), h1 = __float2bfloat16_rn(x[2 * e + 1]);
    hi[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
    lo[e] = pack_bf16x2(x[2 * e] - __bfloat162float(h0), x[2 * e + 1] - __bfloat162float(h1));
  }
  const int jrow = C::ZROW, i0 = (hc >> 1) * 8;
  const int off = (i0 >> 6) * C::SBOX_BYTES + jrow * kRowBytes + ((((i0 & 63) >> 3) ^ (jrow & 7)) << 4);
  uint8_t* img = p.s_image + (size_t)u * C::S_BYTES;
  *reinterpret_cast<uint4*>(img + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  *reinterpret_cast<uint4*>(img + 2 * C::SBOX_BYTES + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

template <int D, bool ROPE>
__device__ void reduce_image(const FusedParams& p) {
  constexpr int TOTAL = (D + (ROPE ? 0 : 1)) * (D / 8);   // chunks of a unit (rotary: the z row goes separately)
  const Sched& s = p.sa;
  const int me = (int)blockIdx.x;
  if (me < s.P * s.U) {
    const int u = me % s.U, c = me / s.U;
    const int lo_i = c * TOTAL / s.P, hi_i = (c + 1) * TOTAL / s.P;
    const int ncol = s.P < (s.tpu + s.Lc - 1) / s.Lc ? s.P : (s.tpu + s.Lc - 1) / s.Lc;
    int r_lo = 0, ntrail = 0;
    if (s.m > 0) {
      const long long ttot = (long long)s.U * s.m;
      r_lo = trailing_cta_of((long long)u * s.m, ttot, s.R);
      ntrail = trailing_cta_of((long long)(u + 1) * s.m - 1, ttot, s.R) - r_lo + 1;
    }
    const int nrec = ncol + ntrail;
    if (hi_i - lo_i <= (int)blockDim.x) {
      reduce_image_chunks<D, ROPE, 1, ROPE ? 6 : 10>(p, u, lo_i + (int)threadIdx.x, hi_i, ncol, r_lo, nrec);
    } else {
      for (int first = lo_i + (int)threadIdx.x; first < hi_i; first += 2 * (int)blockDim.x)
        reduce_image_chunks<D, ROPE, 2, ROPE ? 3 : 6>(p, u, first, hi_i, ncol, r_lo, nrec);
    }
    if (ROPE && D % 8 == 0 && c == 0) reduce_image_zrow<D>(p, u, ncol, r_lo, nrec);
  }
  // The images are read through the async proxy (bulk copy) after the barrier.  (A fence for all of memory, in turn with this: step of 4680 tokens
  // 31.1 and 30.8 us, of 2 x 10800 90.5 and 89.9, forwards level.)
  fence_proxy_async_global();
}

// Eight fp32 values as bf16 hi + lo, sixteen bytes each.
__device__ __forceinline__ void split_hi_lo(const float (&x)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    h[e] = pack_bf16x2(x[2 * e], x[2 * e + 1]);
    l[e] = pack_bf16x2(x[2 * e] - __uint_as_float(h[e] << 16), x[2 * e + 1] - __uint_as_float(h[e] & 0xFFFF0000u));
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// ---------------------------------------------------------------- reduce of a prefill
// All blocks of a cached sequence in one launch: the state that block m's queries see is the cache's, plus the sums of blocks 0..m
// (Eq. 3).  A thread takes 32 bytes of a state row of one head of the cache and walks the blocks: it adds a block's records up in
// their fixed order, adds that to what it has, and leaves the result as the block's operand image (IMAGE) or state.  The records of all
// blocks make one list, of which NR are in flight together (about 148 / heads of them, however they fall on the blocks).  Same sums in
// the same order as a state launch, prefix_states and an apply launch, without the gaps between three launches and with the operands made
// once instead of by every CTA from the states.  Three launches and one, in turn, us: 7 blocks of 4680 tokens, 20 heads of 112 138 and 122, of 10800 298 and 264,
// of 300 34.9 and 22.6 (more beside joins_prefill); 2 entries of 6 blocks of 3040, 35 heads of 64 157 and 144; 7 blocks of 300, 18 heads of 128 39.0 and 22.6.
template <int D, bool IMAGE>
__device__ __forceinline__ void prefix_slice(const FusedParams& p, int& i0, int& i1) {   // this CTA's share of the cache's 32-byte chunks
  const long long tot = (long long)(p.B / p.blocks) * p.H * ((D + 1) * D / 8);
  i0 = (int)(tot * blockIdx.x / gridDim.x);
  i1 = (int)(tot * (blockIdx.x + 1) / gridDim.x);
}

template <int D, bool IMAGE>
__device__ void reduce_prefix(const FusedParams& p) {
  using C = Cfg<D>;
  constexpr int CPR = D / 8, PER_HEAD = (D + 1) * CPR, E4 = (D + 1) * D / 4, REC4 = C::G * E4, NR = 8;
  const Sched& s = p.sa;
  const long long ttot = (long long)s.U * s.m;
  const int ncol = s.P == 0 ? 0 : (s.P < (s.tpu + s.Lc - 1) / s.Lc ? s.P : (s.tpu + s.Lc - 1) / s.Lc);
  int i0, i1;
  prefix_slice<D, IMAGE>(p, i0, i1);
  for (int idx = i0 + (int)threadIdx.x; idx < i1; idx += (int)blockDim.x) {
    const int bh = idx / PER_HEAD, rem = idx - bh * PER_HEAD, j = rem / CPR, c = rem - j * CPR;
    const int b = bh / p.H, h = bh - b * p.H;
    const float4* part4 = reinterpret_cast<const float4*>(p.partials) + (size_t)(h % C::G) * E4 + j * (D / 4) + 2 * c;
    float4* cache4 = reinterpret_cast<float4*>(p.cache) + 2 * (size_t)idx;
    float4 run0 = __ldcg(cache4), run1 = __ldcg(cache4 + 1);
    float4 sum0 = make_float4(0.f, 0.f, 0.f, 0.f), sum1 = sum0;
    // the block whose records come next, its unit, and of its records those that are left
    int m = -1, u = 0, k = 0, nrec = 0, r_lo = 0;
    auto next_block = [&] {
      ++m;
      u = (b * p.blocks + m) * p.HG + h / C::G;
      k = 0;
      nrec = ncol;
      if (s.m > 0) {
        r_lo = trailing_cta_of((long long)u * s.m, ttot, s.R);
        nrec += trailing_cta_of((long long)(u + 1) * s.m - 1, ttot, s.R) - r_lo + 1;
      }
    };
    next_block();
    int done = 0;   // blocks that are complete
    while (done < p.blocks) {
      float4 v[NR][2];
      uint32_t last = 0;   // bit r: record r ends a block
      int n = 0;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (m < p.blocks) {
          const float4* src = part4 + (size_t)(k < ncol ? k * s.U + u : s.P * s.U + r_lo + (k - ncol) + u) * REC4;
          v[r][0] = __ldcg(src);
          v[r][1] = __ldcg(src + 1);
          n = r + 1;
          if (++k == nrec) { last |= 1u << r; next_block(); }
        }
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (r >= n) break;
        add4(sum0, v[r][0]);
        add4(sum1, v[r][1]);
        if (!(last >> r & 1)) continue;
        add4(run0, sum0);
        add4(run1, sum1);
        sum0 = sum1 = make_float4(0.f, 0.f, 0.f, 0.f);
        const int bm = b * p.blocks + done++;
        if (IMAGE) {
          const float x8[8] = {run0.x, run0.y, run0.z, run0.w, run1.x, run1.y, run1.z, run1.w};
          uint4 hi, lo;
          split_hi_lo(x8, hi, lo);
          const int jrow = j < D ? j : C::ZROW, f = c * 8;   // operand row, first key feature
          uint8_t* to = p.s_image + (size_t)(bm * p.H + h) * C::S_BYTES + (f >> 6) * C::SBOX_BYTES + jrow * kRowBytes + ((((f & 63) >> 3) ^ (jrow & 7)) << 4);
          *reinterpret_cast<uint4*>(to) = hi;
          *reinterpret_cast<uint4*>(to + 2 * C::SBOX_BYTES) = lo;
        } else {
          float4* to = reinterpret_cast<float4*>(p.state) + (size_t)(bm * p.H + h) * E4 + j * (D / 4) + 2 * c;
          to[0] = run0;
          to[1] = run1;
        }
      }
    }
    cache4[0] = run0;
    cache4[1] = run1;
  }
  if (IMAGE) fence_proxy_async_global();   // (see reduce_image)
}

// ---------------------------------------------------------------- S operand of the apply pass
// Builds the B operand of the apply MMA for head group (b, hg) from the fp32 state: for every head
// of the group, rows = value features (plus one row for z), K = key features, split into bf16 hi + lo.
template <int D>
__device__ __forceinline__ void build_s_operand(uint8_t* s_op, const float* __restrict__ state, int b, int hg, int H,
                                                int part, int nparts) {
  using C = Cfg<D>;
  constexpr int CPR = D / 8;       // 16-byte chunks per state row
  constexpr int ROWS = D + 1;
  constexpr int TOTAL = C::G * ROWS * CPR;
  constexpr int BATCH = 7;         // chunks whose loads are in flight together (all of a thread's share at d = 112)
  for (int base = part; base < TOTAL; base += BATCH * nparts) {
    float4 lo4[BATCH], hi4[BATCH];
#pragma unroll
    for (int k = 0; k < BATCH; ++k) {
      const int idx = base + k * nparts;
      lo4[k] = hi4[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (idx < TOTAL) {
        const int g = idx / (ROWS * CPR);
        const int rem = idx - g * ROWS * CPR;
        const int j = rem / CPR, c = rem % CPR;
        const int h = hg * C::G + g;
        if (h < H) {
          const float4* src = reinterpret_cast<const float4*>(state + ((size_t)(b * H + h) * ROWS + j) * D + c * 8);
          lo4[k] = __ldcg(src);
          hi4[k] = __ldcg(src + 1);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < BATCH; ++k) {
      const int idx = base + k * nparts;
      if (idx >= TOTAL) break;
      const int g = idx / (ROWS * CPR);
      const int rem = idx - g * ROWS * CPR;
      const int j = rem / CPR, c = rem % CPR;
      const float x[8] = {lo4[k].x, lo4[k].y, lo4[k].z, lo4[k].w, hi4[k].x, hi4[k].y, hi4[k].z, hi4[k].w};
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat16 h0 = __float2bfloat16_rn(x[2 * e]), h1 = __float2bfloat16_rn(x[2 * e + 1]);
        hi[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        lo[e] = pack_bf16x2(x[2 * e] - __bfloat162float(h0), x[2 * e + 1] - __bfloat162float(h1));
      }
      const int jrow = j < D ? g * D + j : C::ZROW + g;  // operand row: value feature, or the head's z row
      const int i0 = g * D + c * 8;                      // first key feature of this chunk
      const int off = (i0 >> 6) * C::SBOX_BYTES + jrow * kRowBytes + ((((i0 & 63) >> 3) ^ (jrow & 7)) << 4);
      *reinterpret_cast<uint4*>(s_op + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(s_op + 2 * C::SBOX_BYTES + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
}

// ---------------------------------------------------------------- lone CTAs
// With few tokens a unit's whole work is done by ONE CTA (kernel instantiation SOLO): the epilogue turns the drained
// accumulators into the apply operand in shared memory where it stands, so that there are no partial records, no grid
// barriers, no reduce and no operand to fetch.  The state MMA has its operands exchanged, A = V^T and B = phi(K), so
// that an accumulator lane is a row of the apply operand (a value feature) and a thread stores sixteen bytes of it at a
// time; with lanes as key features, as the partial records want them, the same step took 20 000 cycles instead of
// 2 500.  z comes from the ReLU warps' fp32 sums, as in the rotary variant.

// Accumulator columns [16 * first, 16 * last) of lane quarter wq (key features; lane = value feature): sums of the four
// accumulators in a fixed order, added (add) to what is staged at `st`, the old state or the tiles before, and left there
// (store) and in the operand (operand).  `st` is copied in at the start and out at the end in one piece (a row per lane
// straight from and to memory took 15 000 cycles, copies of single rows 5 000).  The lanes' rows there are a multiple of 64
// bytes apart, so neighbouring lanes take their four 16-byte pieces in different order: bank conflicts two ways at most.
// Every 64-token tile is drained: an accumulator takes one MMA, the tiles are added up round to nearest, as the grid's
// partial records are.  (One drain at the end made chains of up to eight truncating additions: S of 384 tokens 6.0e-8
// from 64 bits instead of 4.7e-8, with log-normal values 1.2e-7 instead of 4.8e-8.)  The epilogue drains the tiles, and shares
// the columns of the last one with the ReLU warps.
template <int D>
__device__ __forceinline__ void solo_drain(const FusedParams& p, uint8_t* s_op, float* st, uint32_t tmem_base, int wq, int lane, int first, int last,
                                           bool add, bool store, bool operand) {
  using C = Cfg<D>;
  const int i = wq * 32 + lane, g = i / D, il = i - g * D;    // row of the operand, its head of the group, value feature
  const bool live = i < C::FEAT && (int)blockIdx.x % p.HG * C::G + g < p.H;
  float* row = st + (g * (D + 1) + il) * D;
  const int rot = (D == 112 ? lane >> 1 : lane) & 3;
  // x[k] <- x[(k + by) & 3]
  auto turn = [](float4 (&x)[4], int by) {
    const float4 y[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = by & 1 ? y[(k + 1) & 3] : y[k];
    const float4 w[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = by & 2 ? w[(k + 2) & 3] : w[k];
  };
  const uint32_t trow = tmem_base + ((uint32_t)(wq * 32) << 16);
#pragma unroll 1
  for (int cc = first; cc < last && cc * 16 < C::FEAT; ++cc) {
    auto chunk = [&](int c) {   // 16-byte chunk c of the columns in the operand's row of this lane
      const int lc = cc * 2 + c;
      return s_op + (lc >> 3) * C::SBOX_BYTES + i * kRowBytes + (((lc & 7) ^ (i & 7)) << 4);
    };
    if (C::G > 1 && cc * 16 / D != g) {   // blocks across heads are zero (the same for a whole warp)
#pragma unroll
      for (int c = 0; c < 4 && operand; ++c) *reinterpret_cast<uint4*>(chunk(c & 1) + (c >> 1) * 2 * C::SBOX_BYTES) = make_uint4(0, 0, 0, 0);
      continue;
    }
    float4* at = reinterpret_cast<float4*>(row + (C::G == 1 ? cc * 16 : cc * 16 % D));
    uint32_t r[4][16];
#pragma unroll
    for (int a = 0; a < 4; ++a) tmem_ld_x16(trow + a * 128 + cc * 16, r[a]);
    tmem_ld_wait();
    float4 val[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      float f[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        f[e] = live ? __uint_as_float(r[0][4 * x + e]) + __uint_as_float(r[1][4 * x + e]) + __uint_as_float(r[2][4 * x + e]) + __uint_as_float(r[3][4 * x + e]) : 0.f;
      val[x] = make_float4(f[0], f[1], f[2], f[3]);
    }
    if (add && live) {
      float4 old[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) old[k] = at[(k + rot) & 3];
      turn(old, 4 - rot);
#pragma unroll
      for (int x = 0; x < 4; ++x) add4(val[x], old[x]);
    }
    if (operand && i < C::FEAT) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float x8[8] = {val[2 * c].x, val[2 * c].y, val[2 * c].z, val[2 * c].w, val[2 * c + 1].x, val[2 * c + 1].y, val[2 * c + 1].z, val[2 * c + 1].w};
        uint4 hi, lo;
        split_hi_lo(x8, hi, lo);
        *reinterpret_cast<uint4*>(chunk(c)) = hi;
        *reinterpret_cast<uint4*>(chunk(c) + 2 * C::SBOX_BYTES) = lo;
      }
    }
    if (store && live) {
      turn(val, rot);
#pragma unroll
      for (int k = 0; k < 4; ++k) at[(k + rot) & 3] = val[k];
    }
  }
}

// ReLU role: leaves a segment's sums of plain phi(k) in the warp's slot of `slots` and clears them: the four lanes of
// the warp that share a chunk add up in a fixed order, then one of them stores.
__device__ __forceinline__ void leave_z(float* slots, float2 (&zacc)[8], int tr, int lc, bool box1_live) {
  const int w = tr >> 5, r = (tr >> 3) & 3;
  float tot[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) tot[e] = 0.f;
#pragma unroll
  for (int rr = 0; rr < 4; ++rr) {
    const int src = (rr << 3) | (lc ^ ((4 * (w & 1) + rr) & 7));
#pragma unroll
    for (int e = 0; e < 16; ++e) tot[e] += __shfl_sync(0xffffffffu, (e & 1) ? zacc[e >> 1].y : zacc[e >> 1].x, src);
  }
  if (r == 0) {
    float* zp = slots + w * 128;
    *reinterpret_cast<float4*>(zp + 8 * lc) = make_float4(tot[0], tot[1], tot[2], tot[3]);
    *reinterpret_cast<float4*>(zp + 8 * lc + 4) = make_float4(tot[4], tot[5], tot[6], tot[7]);
    if (box1_live) {
      *reinterpret_cast<float4*>(zp + 64 + 8 * lc) = make_float4(tot[8], tot[9], tot[10], tot[11]);
      *reinterpret_cast<float4*>(zp + 64 + 8 * lc + 4) = make_float4(tot[12], tot[13], tot[14], tot[15]);
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) zacc[e] = make_float2(0.f, 0.f);
}

// One feature of the z rows of the apply operand: z in its head's row, zero in the others.
template <int D>
__device__ __forceinline__ void put_z(uint8_t* s_op, int f, float z) {
  using C = Cfg<D>;
  const __nv_bfloat16 hi = __float2bfloat16_rn(z), lo = __float2bfloat16_rn(z - __bfloat162float(hi));
#pragma unroll
  for (int g = 0; g < C::G; ++g) {
    const int jrow = C::ZROW + g;
    uint8_t* at = s_op + (f >> 6) * C::SBOX_BYTES + jrow * kRowBytes + ((((f & 63) >> 3) ^ (jrow & 7)) << 4) + (f & 7) * 2;
    *reinterpret_cast<__nv_bfloat16*>(at) = g == f / D ? hi : __float2bfloat16_rn(0.f);
    *reinterpret_cast<__nv_bfloat16*>(at + 2 * C::SBOX_BYTES) = g == f / D ? lo : __float2bfloat16_rn(0.f);
  }
}

// z of one feature from the sums the warps left in shared memory; the rotary variant's in reduce_image_zrow's association.
template <bool ROPE>
__device__ __forceinline__ float sum_z_slots(const float* slots, int f) {
  auto slot = [&](int w) { return slots[w * 128 + f]; };
  float tree = (slot(0) + slot(1)) + (slot(2) + slot(3));
  if (ROPE) {
    tree += (slot(4) + slot(5)) + (slot(6) + slot(7));
    if (f >= 64) tree += (slot(8) + slot(9)) + (slot(10) + slot(11));
  }
  return tree;
}

// x := 16 bytes at `at` if `live`, loaded into the registers x is in: no branch, no copy and no choice, which would wait for
// the load.
__device__ __forceinline__ void load_in_place(uint4& x, const uint4* at, bool live) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %5, 0;\n"
      "@p ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n"
      "}\n"
      : "+r"(x.x), "+r"(x.y), "+r"(x.z), "+r"(x.w)
      : "l"(at), "r"((int)live));
}

// Rotary variant, state pass: this thread's chunks of the 64 rows of a stage, rows row0 and row0 + 32 of box 0 and row0 of
// box 1 (the epilogue takes the other half of that): plain values to its sums for z, rotated ones back.  All of them are read
// before the first is written.  rows_left: tokens from row0 on; rows beyond the last one hold zeros, and no rotations.
template <int D>
__device__ __forceinline__ void rope_state_rows(uint8_t* k_boxes, const uint8_t* tab, int row0, int pc, int lc, long long rows_left,
                                                float2 (&zacc)[8]) {
  using C = Cfg<D>;
  uint8_t* p0 = k_boxes + row0 * kRowBytes + pc * 16;
  const uint8_t* tb = tab + row0 * C::TAB_ROW;
  uint4 x[3], r[3];   // rows row0 and row0 + 32 of box 0, row0 of box 1
  x[0] = *reinterpret_cast<const uint4*>(p0);
  x[1] = *reinterpret_cast<const uint4*>(p0 + 32 * kRowBytes);
  r[0] = *reinterpret_cast<const uint4*>(tb + C::tab_chunk(0, lc) * 16);
  r[1] = *reinterpret_cast<const uint4*>(tb + 32 * C::TAB_ROW + C::tab_chunk(0, lc) * 16);
  // (d = 112: two lanes of eight have zero padding there, and turn it; without them a branch would part the rows' work)
  x[2] = *reinterpret_cast<const uint4*>(p0 + kBox);
  r[2] = C::SAME_TAB ? r[0] : *reinterpret_cast<const uint4*>(tb + C::tab_chunk(1, lc) * 16);
  if (rows_left <= 32) {
    const uint4 identity = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
    r[1] = identity;
    if (rows_left <= 0) r[0] = r[2] = identity;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    float2 f[4];
    unpack_relu8(x[i], f);
#pragma unroll
    for (int e = 0; e < 4; ++e) zacc[(i == 2 ? 4 : 0) + e] = add2(zacc[(i == 2 ? 4 : 0) + e], f[e]);
    *reinterpret_cast<uint4*>(i == 2 ? p0 + kBox : p0 + i * 32 * kRowBytes) = rotate_pack8(f, r[i]);
  }
}

// Rotary variant, apply pass: this thread's chunks of the 128 rows of a Q tile.  The operand of the numerator is the rotated
// phi(q); the denominator, plain phi(q) . z, is added up over the eight lanes that share a row and left in the row's zero
// padding (features 112..) or in `den`, [G][128].  tab0, tab1: the rotations of its rows for the two boxes (the same
// where box 1 starts a new head); next(i) asks for row i's of the next tile.
//
// The rotary apply pass waits for this role (8 warps): alone on an SM it takes 1450 cycles a tile, with rotations that
// never stall it, where the pass could stream one in 2500.  32 760 tokens, 20 heads of 112, forward: 161 us before the rotations of the
// state pass came through shared memory (its share 84 -> 66 us) and before this function had no branch, copy or choice
// between its rows (77 -> 67 us); 720p 340 -> 282 us, 35 heads of 64 145 -> 137, 18 of 128 150 -> 137.  Not taken: rotations in
// a shared-memory ring beside fewer Q slots (90 to 98 us), sixteen warps of 80 registers (115 us).
template <int D, class Next>
__device__ __forceinline__ void rope_apply_rows(uint8_t* sl, float* den, int row0, int pc, int lc, const float2 (&zc)[8],
                                                const uint4 (&tab0)[kTileApply / 32], const uint4 (&tab1)[kTileApply / 32], Next&& next) {
  using C = Cfg<D>;
  constexpr int HALF = C::SLOT_BYTES / 2;
  uint8_t* p0 = sl + row0 * kRowBytes + pc * 16;
  constexpr int ROWS = kTileApply / 32;
  float dens[ROWS];
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    uint8_t* c0 = p0 + i * 32 * kRowBytes;
    const uint4 x0 = *reinterpret_cast<const uint4*>(c0);
    const uint4 x1 = *reinterpret_cast<const uint4*>(c0 + HALF);
    float2 f[4];
    unpack_relu8(x0, f);
    float2 den2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int e = 0; e < 4; ++e) den2 = fma2(f[e], zc[e], den2);
    *reinterpret_cast<uint4*>(c0) = rotate_pack8(f, tab0[i]);
    float2 den2b = make_float2(0.f, 0.f);   // packed heads: box 1 belongs to other heads than box 0
    unpack_relu8(x1, f);   // (d = 112: padding is turned too, see rope_state_rows; z is zero there)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (C::G == 1) den2 = fma2(f[e], zc[4 + e], den2);
      else den2b = fma2(f[e], zc[4 + e], den2b);
    }
    *reinterpret_cast<uint4*>(c0 + HALF) = rotate_pack8(f, C::SAME_TAB ? tab0[i] : tab1[i]);
    next(i);
    const float dn = dens[i] = den2.x + den2.y;
    // The eight lanes of a row hold one chunk of each box.  Packed heads: box 1 belongs to other heads, and with d = 32 a
    // head is four lanes wide; the first exchange hands one box's sum to the partner lane, so that each half of the lanes
    // reduces one box.
    if (C::G > 1) {
      const int row = row0 + 32 * i;
      const float denb = den2b.x + den2b.y;
      constexpr int XB = C::G == 2 ? 4 : 2;             // lane bit that picks the box after the exchange
      const bool second = (pc & XB) != 0;
      float x = second ? denb : dn;
      x += __shfl_xor_sync(0xffffffffu, second ? dn : denb, XB);
      x += __shfl_xor_sync(0xffffffffu, x, 1);
      if (C::G == 2) x += __shfl_xor_sync(0xffffffffu, x, 2);
      // d = 64: lane 0 of the row has head 0 (box 0), lane 4 head 1.  d = 32: lanes with the same pc / 4 share
      // a head, whose place in its box is lc / 4; lanes 0 and 4 have box 0, lanes 2 and 6 box 1
      if (C::G == 2) {
        if ((pc & 3) == 0) den[(second ? 1 : 0) * kTileApply + row] = x;
      } else {
        if ((pc & 1) == 0) den[((second ? 2 : 0) + (lc >> 2)) * kTileApply + row] = x;
      }
    }
  }
  if (C::G == 1) {
    // One head: four rows over eight lanes.  Each exchange hands half of what a lane has to its partner, so that four
    // shuffles do, not twelve, and lanes 2 i and 2 i + 1 end up with row i.
    const bool b2 = (pc & 4) != 0, b1 = (pc & 2) != 0;
    const float a0 = (b2 ? dens[2] : dens[0]) + __shfl_xor_sync(0xffffffffu, b2 ? dens[0] : dens[2], 4);
    const float a1 = (b2 ? dens[3] : dens[1]) + __shfl_xor_sync(0xffffffffu, b2 ? dens[1] : dens[3], 4);
    float x = (b1 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, b1 ? a0 : a1, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    const int row = row0 + 32 * (pc >> 1);
    if (D == 112) __syncwarp();   // another lane has turned the padding that this row's goes to, and shuffles do not order its store
    if ((pc & 1) == 0) {
      if (D == 112) *reinterpret_cast<float*>(sl + HALF + row * kRowBytes + ((6 ^ (row & 7)) << 4)) = x;   // features 112..119: padding
      else den[row] = x;   // no padding to carry it
    }
  }
}

// Epilogue of an apply tile in slot s: lane quarter wq of accumulator `acc` is divided, rounded and staged in the slot; r:
// accumulator lane = token row of the tile.  The accumulator is handed back as soon as it is read.  (The arguments are what the
// callers' loops have at hand: with ready-made addresses instead the 480p step took 2 % longer.)
template <int D, bool ROPE>
__device__ __forceinline__ void apply_epilogue(uint32_t tmem_base, uint32_t acc, uint8_t* slots, int s, const float* den_rows, int wq, int r, float eps,
                                               uint64_t* c_tempty) {
  using C = Cfg<D>;
  constexpr int SLOT = C::SLOT_BYTES, HALF = SLOT / 2;
  const uint32_t trow = tmem_base + acc * kAccStride + ((uint32_t)(wq * 32) << 16);
  uint8_t* sl = slots + s * SLOT;
  float rinv[C::G];
  if (ROPE) {
    // the ReLU warps left phi(q) . z of this row in the row's padding
    if (D == 112) {
      rinv[0] = 1.0f / (*reinterpret_cast<const float*>(sl + HALF + r * kRowBytes + ((6 ^ (r & 7)) << 4)) + eps);
    } else {
#pragma unroll
      for (int g = 0; g < C::G; ++g) rinv[g] = 1.0f / (den_rows[(s * C::G + g) * kTileApply + r] + eps);
    }
  } else {
    uint32_t dn[4];
    tmem_ld_x4(trow + C::ZROW, dn);
    tmem_ld_wait();
#pragma unroll
    for (int g = 0; g < C::G; ++g) rinv[g] = 1.0f / (__uint_as_float(dn[g]) + eps);  // eps added once, after the dot product
  }
#pragma unroll
  for (int cc = 0; cc < 4; ++cc) {
    if (cc * 32 >= C::FEAT) break;
    uint32_t v[32];
    tmem_ld_x32(trow + cc * 32, v);
    tmem_ld_wait();
    if (cc == 3 || (cc + 1) * 32 >= C::FEAT) {  // last read of this accumulator: hand it back to the MMA warp
      tcgen05_fence_before();
      mbar_arrive(&c_tempty[acc]);
    }
    const float ri = rinv[(cc * 32) / D < C::G ? (cc * 32) / D : 0];
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
      const int lc = cc * 4 + q4;  // logical 16-byte chunk of the 256-byte padded row
      if (lc * 8 >= C::FEAT) break;
      uint4 pk;
      pk.x = pack_bf16x2(__uint_as_float(v[q4 * 8 + 0]) * ri, __uint_as_float(v[q4 * 8 + 1]) * ri);
      pk.y = pack_bf16x2(__uint_as_float(v[q4 * 8 + 2]) * ri, __uint_as_float(v[q4 * 8 + 3]) * ri);
      pk.z = pack_bf16x2(__uint_as_float(v[q4 * 8 + 4]) * ri, __uint_as_float(v[q4 * 8 + 5]) * ri);
      pk.w = pack_bf16x2(__uint_as_float(v[q4 * 8 + 6]) * ri, __uint_as_float(v[q4 * 8 + 7]) * ri);
      *reinterpret_cast<uint4*>(sl + (lc >> 3) * HALF + r * kRowBytes + (((lc & 7) ^ (r & 7)) << 4)) = pk;
    }
  }
}

// ============================================================================ the kernel
// SOLO: lone CTAs.  IMAGE: the reduce leaves operand images and the apply pass fetches them (p.s_image).  Both are decided
// on the host, and each form is a kernel of its own: the rotary one has no registers to spare, and with the slice reduce that
// it does not take compiled into it (even out of line) a read-only rotary step of 4680 tokens took 45.0 us instead of 43.1.
// PREFIX: a prefill of several blocks (p.blocks, p.cache), the reduce is reduce_prefix.
template <int D, bool ROPE, bool SOLO, bool IMAGE, bool PREFIX = false>
__global__ void __launch_bounds__(Roles<ROPE>::THREADS, 1)
umma_fused_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                  const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o,
                  const __grid_constant__ FusedParams p) {
  static_assert(!IMAGE || (Cfg<D>::G == 1 && !SOLO), "operand images are of one-head units in a grid");
  using C = Cfg<D>;
  using R = Roles<ROPE>;
  // TAB: the state pass has its rotations in shared memory.  (Lone CTAs have no room for them and fetch them into registers.)
  constexpr bool TAB = ROPE && !SOLO;
  // QT: phi(Q) is an operand in tensor memory, beside the accumulator of its tile.  Of the 260 KB that a tile of 128 rows moves through shared
  // memory that takes out 84 (the clamped rows back, and both MMAs' reads of them): time where a tile is waited for, power where the
  // chip is at its cap (1000 W, 1.5 to 1.6 GHz: forwards of 32 760 tokens and more).  Without and with, in turn, us: step of 4680 tokens 31.1 and 30.8, of
  // 2 x 10800 90.7 and 89.9, forward of 75 600 tokens, 35 heads of 64 252.7 and 249.4; 20 heads of 112 level (32 760 tokens 124.8 and 124.2, 75 600 266 and
  // 267, runs of one side differ by 1 to 2 %); same bits.  (Lone CTAs: their accumulators take
  // all columns up to the first Q tile.  Rotary: the rotated rows come eight lanes to a row.)
  constexpr bool QT = !ROPE && !SOLO;
  constexpr uint32_t QT_COL = 160;         // behind the accumulator's columns
  static_assert(!QT || (C::NAPPLY <= QT_COL && QT_COL + C::FEAT / 2 <= kAccStride), "columns of tensor memory");
  constexpr int NSA = SOLO ? 4 : ROPE ? C::ROPE_STAGES : C::STATE_STAGES;
  constexpr int STAGE = SOLO ? C::SOLO_STAGE_BYTES : ROPE ? C::ROPE_STAGE_BYTES : C::STAGE_BYTES;
  constexpr int KOFF = SOLO || ROPE ? 2 * kBox : C::KOFF;
  constexpr int TOFF = 4 * kBox;
  constexpr int NSC = SOLO ? C::SOLO_SLOTS : C::APPLY_SLOTS;
  constexpr int DATA = SOLO ? C::SOLO_DATA : C::DATA_BYTES;
  constexpr int SLOT = C::SLOT_BYTES;
  constexpr int HALF = SLOT / 2;  // one 64-feature box of 128 tokens
  constexpr uint32_t IDESC_A = make_idesc_bf16(128, SOLO || ROPE ? 128 : C::NSTATE, true, true);
  constexpr int ACCS = SOLO || ROPE ? 4 : C::STATE_ACCS, ACC_STRIDE = SOLO || ROPE ? 128 : C::STATE_ACC_STRIDE;
  constexpr uint32_t IDESC_C = make_idesc_bf16(128, C::NAPPLY, false, false);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* s_op = smem;                    // apply pass: S operand ...
  uint8_t* slots = smem + C::S_BYTES;      // ... and the Q/O slots; the state pass stages cover both
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + DATA);
  // state pass
  uint64_t* a_full = bars;                 // TMA landed
  uint64_t* a_ready = a_full + NSA;        // ReLU pass done
  uint64_t* a_empty = a_ready + NSA;       // MMAs that read the stage are complete
  uint64_t* a_tfull = a_empty + NSA;       // the segment's accumulators are complete
  uint64_t* a_tempty = a_tfull + 2;        // ... and drained by the epilogue
  uint64_t* a_done = a_tempty + 2;         // every MMA of the state pass is complete: stages are free
  // apply pass
  uint64_t* c_full = a_done + 1;           // Q tile landed
  uint64_t* c_ready = c_full + NSC;        // ReLU pass done
  uint64_t* c_empty = c_ready + NSC;       // O tile read out by its TMA store: slot reusable
  uint64_t* c_staged = c_empty + NSC;      // the 128 epilogue threads have written their O rows
  uint64_t* c_tfull = c_staged + NSC;      // [2] accumulator complete
  uint64_t* c_tempty = c_tfull + 2;        // [2] accumulator drained
  uint64_t* s_ready = c_tempty + 2;        // S operand of the current segment is in shared memory
  uint64_t* seg_done = s_ready + 1;        // every MMA of the finished segment is complete
  uint64_t* z_left = seg_done + 1;         // lone CTAs: every warp's share of z is in shared memory ...
  uint64_t* z_done = z_left + 1;           // ... and (rotary) z itself
  uint64_t* st_full = z_done + 1;          // lone CTAs: the old state is in shared memory
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(st_full + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  float* den_rows = reinterpret_cast<float*>(smem + DATA + C::BAR_BYTES);   // [NSC][G][128]: rotary variant, every head dim but 112
  static_assert((3 * NSA + 5 + 4 * NSC + 9) * 8 + 8 <= C::BAR_BYTES, "barrier block too small");
  // lone CTAs: [kZSlots][128] sums of plain phi(k), then z, then the state, behind the stages and the slots
  float* z_slots = reinterpret_cast<float*>(smem + C::SOLO_Z);
  float* z_row = z_slots + kZParts;
  float* st = reinterpret_cast<float*>(smem + C::SOLO_STATE);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Work wa = p.do_state ? work_of(p.sa, blockIdx.x) : work_of(p.sa, 0x7fffffff);
  const Work wc = p.do_apply ? work_of(p.sc, blockIdx.x) : work_of(p.sc, 0x7fffffff);

  // generation of the grid-barrier word before this launch's first barrier (it cannot move until every CTA, this
  // one included, has arrived): read once, early, so that an arrival needs no answer from memory
  unsigned gen0 = 0;
  if (!SOLO && threadIdx.x == 0 && p.do_state) gen0 = ld_acquire_gpu(&p.ctrl->barrier[0]) >> 16;
  if (threadIdx.x == 0) {
    if (!SOLO && blockIdx.x == 0 && p.do_state) grid_barrier_preset(p.ctrl);   // for the first grid barrier
    for (int s = 0; s < NSA; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_ready[s], R::RELU_THREADS + (ROPE ? 128 : 0)); mbar_init(&a_empty[s], 1); }
    mbar_init(a_tfull, 1);
    mbar_init(a_tempty, 128);
    mbar_init(a_done, 1);
    for (int s = 0; s < NSC; ++s) {
      mbar_init(&c_full[s], 1); mbar_init(&c_ready[s], R::RELU_THREADS); mbar_init(&c_empty[s], 1); mbar_init(&c_staged[s], 128);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(&c_tfull[b], 1); mbar_init(&c_tempty[b], 128); }
    mbar_init(s_ready, R::RELU_THREADS + 128);
    mbar_init(seg_done, 128);
    if (SOLO) { mbar_init(z_left, R::RELU_THREADS + (ROPE ? 128 : 0)); mbar_init(z_done, R::RELU_THREADS); mbar_init(st_full, 1); }
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tensormap(&map_k);
    prefetch_tensormap(&map_v);
    prefetch_tensormap(&map_q);
    prefetch_tensormap(&map_o);
  }
  if (!SOLO && !ROPE && C::ONES_BOX && wa.f1 > wa.f0) {
    // the constant "ones" chunk of every stage: value columns 128..191 of B, of which column 128 is 1
    for (int idx = threadIdx.x; idx < NSA * (kBox / 16); idx += R::THREADS) {
      const int s = idx / (kBox / 16), c = idx % (kBox / 16);
      const int row = c >> 3, phys = c & 7;
      uint4 val = make_uint4(0, 0, 0, 0);
      if ((phys ^ (row & 7)) == 0) val.x = 0x3F80u;  // bf16 1.0 in element 0 of logical chunk 0
      *reinterpret_cast<uint4*>(smem + s * STAGE + 2 * kBox + c * 16) = val;
    }
    fence_proxy_async_smem();
  }
  if (SOLO) wait_for_prior_grids();
  if (warp == 1) { tmem_alloc(tmem_holder, kTmemCols); tmem_relinquish(); }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  if (SOLO) let_next_grid_start();
  const uint32_t tmem_base = *tmem_holder;

  // apply-pass producer state lives across the grid barriers (the first tiles are fetched before them)
  TileWalk cw(wc);
  uint32_t c_it = 0;
  auto load_q_tile = [&]() -> bool {
    const int s = c_it % NSC;
    if (!mbar_wait(&c_empty[s], ((c_it / NSC) & 1) ^ 1, abort_flag)) return false;
    const int u = cw.unit(), b = u / p.HG, hg = u % p.HG;
    uint8_t* sl = slots + s * SLOT;
    mbar_arrive_expect_tx(&c_full[s], SLOT);
    int c0, c1;
    box_coords<D>(0, hg, c0, c1);
    tma_load_4d(sl, &map_q, &c_full[s], c0, c1, cw.tile() * kTileApply, b);
    box_coords<D>(1, hg, c0, c1);
    tma_load_4d(sl + HALF, &map_q, &c_full[s], c0, c1, cw.tile() * kTileApply, b);
    cw.next();
    ++c_it;
    return true;
  };

  // ==================================================================== state pass
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      for (TileWalk t(wa); !t.done(); t.next(), ++it) {
        const int s = it % NSA;
        if (!mbar_wait(&a_empty[s], ((it / NSA) & 1) ^ 1, abort_flag)) break;
        const int u = t.unit(), b = u / p.HG, hg = u % p.HG;
        uint8_t* st = smem + s * STAGE;
        if (TAB) {
          const long long n = (long long)t.tile() * kTileState, left = p.N - n;
          const uint32_t bytes = (left < kTileState ? (uint32_t)left : (uint32_t)kTileState) * C::TAB_ROW;
          mbar_arrive_expect_tx(&a_full[s], 4 * kBox + bytes);
          bulk_load(st + TOFF, p.rope + n * (D / 8), bytes, &a_full[s]);
        } else {
          mbar_arrive_expect_tx(&a_full[s], 4 * kBox);
        }
        int c0, c1;
        box_coords<D>(0, hg, c0, c1);
        tma_load_4d(st + KOFF, &map_k, &a_full[s], c0, c1, t.tile() * kTileState, b);
        tma_load_4d(st, &map_v, &a_full[s], c0, c1, t.tile() * kTileState, b);
        box_coords<D>(1, hg, c0, c1);
        tma_load_4d(st + KOFF + kBox, &map_k, &a_full[s], c0, c1, t.tile() * kTileState, b);
        tma_load_4d(st + kBox, &map_v, &a_full[s], c0, c1, t.tile() * kTileState, b);
      }
      // Q does not depend on the state: fill the slots as soon as every MMA of this pass is complete (the
      // stages are free then).  Asking for tiles earlier or further ahead with TMA prefetches into L2
      // measured slower at every distance tried (0-24 tiles).
      if (wc.f1 > wc.f0 && mbar_wait(a_done, 0, abort_flag)) {
        while (!cw.done() && c_it < (uint32_t)NSC)
          if (!load_q_tile()) break;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      uint32_t it = 0, seg = 0, n_mma = 0;
      bool ok = true;
      for (TileWalk t(wa); !t.done() && ok; t.next(), ++it) {
        const int s = it % NSA;
        const bool seg_first = t.seg_first();
        if (SOLO || seg_first) { ok = mbar_wait(a_tempty, (seg & 1) ^ 1, abort_flag); n_mma = 0; }
        if (ok) ok = mbar_wait(&a_ready[s], (it / NSA) & 1, abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        const uint32_t st = smem_u32(smem + s * STAGE);
#pragma unroll
        for (int kk = 0; kk < kTileState / 16; ++kk, ++n_mma) {
          const uint64_t a = make_smem_desc_sw128(st + KOFF + kk * 2048, kBox, 1024);  // phi(K)^T, MN-major
          const uint64_t bq = make_smem_desc_sw128(st + kk * 2048, kBox, 1024);           // [V | 1], MN-major
          const uint32_t d_tmem = tmem_base + (n_mma % ACCS) * ACC_STRIDE;
          umma_bf16(d_tmem, SOLO ? bq : a, SOLO ? a : bq, IDESC_A, n_mma < (uint32_t)ACCS ? 0u : 1u);  // first use of each: overwrite
        }
        umma_commit(&a_empty[s]);
        if (SOLO || t.seg_last()) { umma_commit(a_tfull); ++seg; }
      }
      if (it > 0) umma_commit(a_done); else mbar_arrive(a_done);
    }
  } else if (warp < R::EPI_WARP0) {
    // ------------------------------------------------------------ ReLU pass over the K boxes
    const int tr = threadIdx.x - kReluThread0;
    uint32_t it = 0;
    // rotary variant: this thread's 16-byte column holds logical chunk lc of every row it touches
    const int row0 = tr >> 3, pc = tr & 7, lc = pc ^ (row0 & 7);
    const bool box1_live = 64 + lc * 8 < C::FEAT;
    float2 zacc[8];  // sums of the plain phi(k) over the segment: features 8*lc.. of box 0, 64 + 8*lc.. of box 1
#pragma unroll
    for (int e = 0; e < 8; ++e) zacc[e] = make_float2(0.f, 0.f);
    // Lone CTAs: the rotations of a row do not depend on K; they are fetched one stage ahead, each register reloaded
    // for the next stage right after its use, so that their latency is off the stage's critical path.
    // Of the second K box these warps take the first 32 token rows of a stage; the epilogue warps, idle until the
    // segment's accumulators are complete, take the other 32 (this role is what the pass waits for).
    uint4 tab0[kTileState / 32], tab1[1];
    const uint4* const rope = SOLO && ROPE ? behind_wait(p.rope) : p.rope;
    auto fetch_rot = [&](int tile, int i) {
      const long long n = (long long)tile * kTileState + row0 + 32 * i;
      tab0[i] = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
      if (i == 0) tab1[0] = tab0[i];
      if (n < p.N) {
        tab0[i] = __ldg(rope + n * (D / 8) + C::tab_chunk(0, lc));
        if (i == 0) {
          if (C::SAME_TAB) tab1[0] = tab0[0];
          else if (box1_live) tab1[0] = __ldg(rope + n * (D / 8) + C::tab_chunk(1, lc));
        }
      }
    };
    // lone CTAs: z from the warps' sums, to memory and (plain) into the operand or (rotary) where this role finds it.
    // A warp whose wait ran out does not report its share of the operand: then nothing is applied and no state leaves.
    auto finish_z = [&]() {
      mbar_arrive(z_left);
      bool ok = mbar_wait(z_left, 0, abort_flag);               // every warp's sums are in shared memory
      if (!ROPE) ok = ok && mbar_wait(a_done, 0, abort_flag);   // the operand lies where the stages were
      const int f = tr, g = f / D, h = ((int)blockIdx.x % p.HG) * C::G + g;
      if (p.accumulate) ok = ok && mbar_wait(st_full, 0, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) return;
      if (f < C::FEAT) {
        float z = sum_z_slots<ROPE>(z_slots, f);
        float* at = st + (g * (D + 1) + D) * D + (f - g * D);
        if (p.accumulate && h < p.H) z += *at;
        if (p.write_state) *at = z;
        if (ROPE) z_row[f] = z;
        else if (p.do_apply) put_z<D>(s_op, f, z);
      }
      if (ROPE) {
        mbar_arrive(z_done);
        ok = mbar_wait(z_done, 0, abort_flag);
      }
      // this role's share of the drain
      // (a_done: the last tile's accumulators, and the drain of the tile before it has come to its end; looking for that at
      // a_tempty makes this thread see what the epilogue left at st)
      const int tiles = (int)(wa.f1 - wa.f0);
      ok = ok && mbar_wait(a_done, 0, abort_flag);
      if (tiles > 1) ok = ok && mbar_wait(a_tempty, tiles & 1, abort_flag);
      if (!__all_sync(0xffffffffu, ok)) return;
      tcgen05_fence_after();
      const int half = tr >> 7;   // (rotary variant: two warps of this role to a lane quarter)
      const int c0 = ROPE ? 3 + 3 * half : 4, c1 = ROPE && !half ? 6 : 8;
      solo_drain<D>(p, s_op, st, tmem_base, warp & 3, lane, c0, c1, p.accumulate || tiles > 1, p.write_state, p.do_apply);
      tcgen05_fence_before();
      fence_proxy_async_smem();
      mbar_arrive(s_ready);
    };
    if (ROPE && SOLO) {
      TileWalk t0(wa);
      if (!t0.done()) {
#pragma unroll
        for (int i = 0; i < kTileState / 32; ++i) fetch_rot(t0.tile(), i);
      }
    }
    for (TileWalk t(wa); !t.done(); t.next(), ++it) {
      const int s = it % NSA;
      uint8_t* st = smem + s * STAGE;
      if (TAB) {
        if (!__all_sync(0xffffffffu, mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag))) break;  // leave as a whole warp
        rope_state_rows<D>(st + KOFF, st + TOFF, row0, pc, lc, p.N - (long long)t.tile() * kTileState - row0, zacc);
        fence_proxy_async_smem();
        mbar_arrive(&a_ready[s]);
        if (t.seg_last())
          leave_z(p.partials + (size_t)t.record() * (C::G * (D + 1) * D + kZParts) + C::G * (D + 1) * D, zacc, tr, lc, box1_live);
        continue;
      }
      if (ROPE) {
        TileWalk tn = t;
        tn.next();
        if (!__all_sync(0xffffffffu, mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag))) break;  // leave as a whole warp
        uint8_t* p0 = st + KOFF + row0 * kRowBytes + pc * 16;
#pragma unroll
        for (int i = 0; i < kTileState / 32; ++i) {
          float2 f[4];
          uint4* c0 = reinterpret_cast<uint4*>(p0 + i * 32 * kRowBytes);
          unpack_relu8(*c0, f);
#pragma unroll
          for (int e = 0; e < 4; ++e) zacc[e] = add2(zacc[e], f[e]);
          *c0 = rotate_pack8(f, tab0[i]);
          if (i == 0 && box1_live) {
            uint4* c1 = reinterpret_cast<uint4*>(p0 + kBox);
            unpack_relu8(*c1, f);
#pragma unroll
            for (int e = 0; e < 4; ++e) zacc[4 + e] = add2(zacc[4 + e], f[e]);
            *c1 = rotate_pack8(f, tab1[0]);
          }
          if (!tn.done()) fetch_rot(tn.tile(), i);
        }
        fence_proxy_async_smem();
        mbar_arrive(&a_ready[s]);
        if (t.seg_last()) {
          leave_z(z_slots, zacc, tr, lc, box1_live);
          finish_z();
        }
        continue;
      }
      if (SOLO) {
        if (!__all_sync(0xffffffffu, mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag))) break;  // leave as a whole warp
        relu_sum_pass<C::FEAT, kTileState>(st + KOFF, st + KOFF + kBox, tr, zacc);
        fence_proxy_async_smem();
        mbar_arrive(&a_ready[s]);
        if (t.seg_last()) {
          leave_z(z_slots, zacc, tr, lc, box1_live);
          finish_z();
        }
        continue;
      }
      if (!mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag)) break;
      relu_pass<C::FEAT, kTileState>(st + KOFF, st + KOFF + kBox, tr);
      if (!C::ONES_BOX && tr < kTileState) {
        // value column 112 := 1 (logical chunk 6 of the second V box, element 0), so z is accumulator column 112
        *reinterpret_cast<uint16_t*>(st + kBox + tr * kRowBytes + ((6 ^ (tr & 7)) << 4)) = 0x3F80u;
      }
      fence_proxy_async_smem();
      mbar_arrive(&a_ready[s]);
    }
  } else if (warp < R::STORE_WARP) {
    // ------------------------------------------------------------ epilogue: accumulator -> partial record
    const int wq = warp & 3;
    const int i = wq * 32 + lane;           // accumulator lane = key feature within the group
    const int g = i / D, il = i % D;        // head within the group, feature within the head
    uint32_t seg = 0;
    // rotary variant: token rows 32..63 of the second K box of every stage (see the ReLU role); thread te owns
    // the 16-byte column position pch of rows 32 + row0h + 16 j, which holds logical chunk lch in all of them
    const int te = threadIdx.x - R::EPI_THREAD0;
    const int row0h = te >> 3, pch = te & 7, lch = pch ^ (row0h & 7);
    const bool h_live = 64 + lch * 8 < C::FEAT;
    float2 zh[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) zh[e] = make_float2(0.f, 0.f);
    uint4 tabh[2];
    const uint4* const rope = SOLO && ROPE ? behind_wait(p.rope) : p.rope;
    auto fetch_roth = [&](int tile, int j) {
      const long long n = (long long)tile * kTileState + 32 + row0h + 16 * j;
      tabh[j] = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
      if (h_live && n < p.N) tabh[j] = __ldg(rope + n * (D / 8) + C::tab_chunk(1, lch));
    };
    if (ROPE && SOLO) {
      TileWalk t0(wa);
      if (!t0.done()) { fetch_roth(t0.tile(), 0); fetch_roth(t0.tile(), 1); }
    }
    uint32_t it = 0;
    for (TileWalk t(wa); !t.done(); t.next(), ++it) {
      if (ROPE) {
        const int s = it % NSA;
        TileWalk tn = t;
        tn.next();
        if (!__all_sync(0xffffffffu, mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag))) break;  // leave as a whole warp
        uint8_t* p1 = smem + s * STAGE + KOFF + kBox + (32 + row0h) * kRowBytes + pch * 16;
        if (TAB) {   // this tile's, from its stage
          const uint8_t* tb = smem + s * STAGE + TOFF + (32 + row0h) * C::TAB_ROW + C::tab_chunk(1, lch) * 16;
          const long long rows_left = p.N - (long long)t.tile() * kTileState - 32 - row0h;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            tabh[j] = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
            if (h_live && rows_left > 16 * j) tabh[j] = *reinterpret_cast<const uint4*>(tb + j * 16 * C::TAB_ROW);
          }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (h_live) {
            float2 f[4];
            uint4* c1 = reinterpret_cast<uint4*>(p1 + j * 16 * kRowBytes);
            unpack_relu8(*c1, f);
#pragma unroll
            for (int e = 0; e < 4; ++e) zh[e] = add2(zh[e], f[e]);
            *c1 = rotate_pack8(f, tabh[j]);
          }
          if (SOLO && !tn.done()) fetch_roth(tn.tile(), j);
        }
        fence_proxy_async_smem();
        mbar_arrive(&a_ready[s]);
        if (t.seg_last()) {
          // this warp's share of the segment's z: the four lanes that share a chunk add up in a fixed order
          const int rq = (te >> 3) & 3;
          float tot[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) tot[e] = 0.f;
#pragma unroll
          for (int rr = 0; rr < 4; ++rr) {
            const int src = (rr << 3) | (lch ^ ((4 * ((te >> 5) & 1) + rr) & 7));
#pragma unroll
            for (int e = 0; e < 8; ++e) tot[e] += __shfl_sync(0xffffffffu, (e & 1) ? zh[e >> 1].y : zh[e >> 1].x, src);
          }
          if (rq == 0 && h_live) {
            float* zp = (SOLO ? z_slots : p.partials + (size_t)t.record() * (C::G * (D + 1) * D + kZParts) + C::G * (D + 1) * D) + (8 + (te >> 5)) * 128;
            *reinterpret_cast<float4*>(zp + 64 + 8 * lch) = make_float4(tot[0], tot[1], tot[2], tot[3]);
            *reinterpret_cast<float4*>(zp + 64 + 8 * lch + 4) = make_float4(tot[4], tot[5], tot[6], tot[7]);
          }
          if (SOLO) mbar_arrive(z_left);
#pragma unroll
          for (int e = 0; e < 4; ++e) zh[e] = make_float2(0.f, 0.f);
        }
      }
      if (!SOLO && !t.seg_last()) continue;
      bool ok = mbar_wait(a_tfull, seg & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tcgen05_fence_after();
      if (SOLO) {
        const bool last = t.seg_last();
        if (p.accumulate && it == 0 && !__all_sync(0xffffffffu, mbar_wait(st_full, 0, abort_flag))) break;
        solo_drain<D>(p, s_op, st, tmem_base, wq, lane, 0, !last ? 8 : ROPE ? 3 : 4, p.accumulate || it > 0, !last || p.write_state, last && p.do_apply);
        if (last) fence_proxy_async_smem();   // the operand is read by the MMAs of the apply pass
        tcgen05_fence_before();
        mbar_arrive(last ? s_ready : a_tempty);
        ++seg;
        continue;
      }
      const int u = t.unit(), hg = u % p.HG;
      const int h = hg * C::G + g;
      const bool live = i < C::FEAT && h < p.H;
      // record of this (CTA, unit) segment: G consecutive head-states in the library's layout
      float* out = p.partials + (size_t)t.record() * (C::G * (D + 1) * D + (ROPE ? kZParts : 0)) + (size_t)g * ((D + 1) * D);
      const uint32_t trow = tmem_base + ((uint32_t)(wq * 32) << 16);
#pragma unroll 1
      for (int cc = 0; cc < 4; ++cc) {
        // the accumulators are added in a fixed order (round to nearest)
        float sum[32];
        {
          uint32_t r[32];
          tmem_ld_x32(trow + cc * 32, r);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 32; ++x) sum[x] = __uint_as_float(r[x]);
        }
#pragma unroll 1
        for (int a = 1; a < ACCS; ++a) {
          uint32_t r[32];
          tmem_ld_x32(trow + a * ACC_STRIDE + cc * 32, r);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 32; ++x) sum[x] += __uint_as_float(r[x]);
        }
        if (live) {
#pragma unroll
          for (int x = 0; x < 32; ++x) {
            const int j = cc * 32 + x;             // value feature within the group
            const int jl = j - g * D;
            if (jl >= 0 && jl < D) out[(size_t)jl * D + il] = sum[x];
            if (!C::ONES_BOX && !ROPE && j == C::ZCOL) out[(size_t)D * D + il] = sum[x];  // (rotary: z comes from the ReLU warps)
          }
        }
      }
      if (C::ONES_BOX && !ROPE) {   // (rotary: z comes from the ReLU warps)
        float zsum = 0.f;
#pragma unroll 1
        for (int a = 0; a < C::STATE_ACCS; ++a) {
          uint32_t zr[4];
          tmem_ld_x4(trow + a * C::STATE_ACC_STRIDE + C::ZCOL, zr);
          tmem_ld_wait();
          zsum = a == 0 ? __uint_as_float(zr[0]) : zsum + __uint_as_float(zr[0]);
        }
        if (live) out[(size_t)D * D + il] = zsum;
      }
      tcgen05_fence_before();
      mbar_arrive(a_tempty);
      ++seg;
    }
  } else if (SOLO) {
    // ------------------------------------------------------------ store warp: the state in, and out again
    if (lane == 0) {
      const int b = (int)blockIdx.x / p.HG, h0 = ((int)blockIdx.x % p.HG) * C::G, heads = p.H - h0 < C::G ? p.H - h0 : C::G;
      const size_t at = (size_t)(b * p.H + h0) * ((D + 1) * D);
      const uint32_t bytes = heads * (D + 1) * D * 4;
      if (p.accumulate) {
        mbar_arrive_expect_tx(st_full, bytes);
        bulk_load(st, p.state_base + at, bytes, st_full);
      }
      if (p.write_state && mbar_wait(s_ready, 0, abort_flag)) {
        bulk_store(p.state + at, st, bytes);
        tma_store_commit();
      }
    }
    __syncwarp();
  } else if (PREFIX) {
    // ------------------------------------------------------------ store warp (idle in this pass): the cache into L2, as below
    if (__all_sync(0xffffffffu, mbar_wait(a_done, 0, abort_flag))) {
      int i0, i1;
      prefix_slice<D, IMAGE>(p, i0, i1);
      const char* base = reinterpret_cast<const char*>(p.cache) + (size_t)i0 * 32;
      for (int off = lane * 128; off < (i1 - i0) * 32; off += 32 * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(base + off) : "memory");
    }
  } else if (IMAGE && p.accumulate && p.do_state && (int)blockIdx.x < p.sa.P * p.sa.U) {
    // ------------------------------------------------------------ store warp (idle in this pass)
    // A cached step adds to the old state, which the K, V stream has pushed out of L2 since the last step:
    // once this CTA's loads are all issued, ask for its share of it (reduce_image's split), so that the
    // reduce finds it in L2 instead of waiting for DRAM between the two grid barriers.
    if (__all_sync(0xffffffffu, mbar_wait(a_done, 0, abort_flag))) {
      constexpr int TOTAL = (D + (ROPE ? 0 : 1)) * (D / 8);
      const int u = (int)blockIdx.x % p.sa.U, c = (int)blockIdx.x / p.sa.U;
      const int lo_i = c * TOTAL / p.sa.P, hi_i = (c + 1) * TOTAL / p.sa.P;
      const char* base = reinterpret_cast<const char*>(p.state_base + (size_t)u * ((D + 1) * D)) + (size_t)lo_i * 32;
      for (int off = lane * 128; off < (hi_i - lo_i) * 32; off += 32 * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(base + off) : "memory");
    }
  }

  // ==================================================================== reduce
  if (!SOLO && p.do_state) {
    grid_barrier(p.ctrl, abort_flag, p.do_apply != 0, gen0);
    if (!*abort_flag) {
      if constexpr (PREFIX) reduce_prefix<D, IMAGE>(p);
      else if constexpr (IMAGE) reduce_image<D, ROPE>(p);
      else reduce_slice<D, ROPE>(p);
    }
    if (p.do_apply) grid_barrier(p.ctrl, abort_flag, false, gen0 + 1);
  }
  if (!SOLO && C::G > 1 && wc.f1 > wc.f0) {
    // cross-head blocks of the packed S operand are never written by a head: they must read as zero
    for (int idx = threadIdx.x; idx < C::S_BYTES / 16; idx += R::THREADS)
      *reinterpret_cast<uint4*>(s_op + idx * 16) = make_uint4(0, 0, 0, 0);
    __syncthreads();
  }

  // ==================================================================== apply pass
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer: the remaining Q tiles
    if (lane == 0) {
      while (!cw.done())
        if (!load_q_tile()) break;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      uint32_t it = 0, seg = 0;
      bool ok = true;
      for (TileWalk t(wc); !t.done() && ok; t.next(), ++it) {
        const int s = it % NSC;
        if (t.seg_first()) { ok = mbar_wait(s_ready, seg & 1, abort_flag); ++seg; }
        const uint32_t acc = it & 1;
        if (ok) ok = mbar_wait(&c_tempty[acc], ((it >> 1) & 1) ^ 1, abort_flag);
        if (ok) ok = mbar_wait(&c_ready[s], (it / NSC) & 1, abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        const uint32_t d_tmem = tmem_base + acc * kAccStride;
        const uint32_t a0 = smem_u32(slots + s * SLOT);
        const uint32_t b0 = smem_u32(s_op);
#pragma unroll
        for (int k = 0; k < C::KSTEPS; ++k) {
          const uint32_t koff = (k >> 2) * HALF + (k & 3) * 32;
          const uint32_t boff = (k >> 2) * C::SBOX_BYTES + (k & 3) * 32;
          const uint64_t a = make_smem_desc_sw128(a0 + koff, 16, 1024);                           // phi(Q), K-major
          const uint64_t bh = make_smem_desc_sw128(b0 + boff, 16, 1024);                          // S hi
          const uint64_t bl = make_smem_desc_sw128(b0 + 2 * C::SBOX_BYTES + boff, 16, 1024);      // S lo
          if (QT) {
            umma_bf16_ts(d_tmem, d_tmem + QT_COL + k * 8, bh, IDESC_C, k == 0 ? 0u : 1u);
            umma_bf16_ts(d_tmem, d_tmem + QT_COL + k * 8, bl, IDESC_C, 1u);
          } else {
            umma_bf16(d_tmem, a, bh, IDESC_C, k == 0 ? 0u : 1u);
            umma_bf16(d_tmem, a, bl, IDESC_C, 1u);
          }
        }
        umma_commit(&c_tfull[acc]);
      }
    }
  } else if (warp < R::EPI_WARP0) {
    // ------------------------------------------------------------ ReLU pass over Q tiles (+ half of the S build)
    const int tr = threadIdx.x - kReluThread0;
    uint32_t it = 0, seg = 0;
    bool ok = true;
    // rotary variant: this thread's 16-byte column holds logical chunk lc of every row it touches
    const int row0 = tr >> 3, pc = tr & 7, lc = pc ^ (row0 & 7);
    const bool box1_live = 64 + lc * 8 < C::FEAT;
    float2 zc[8];  // the segment's z at this thread's features (8*lc.. of box 0, 64 + 8*lc.. of box 1)
#pragma unroll
    for (int e = 0; e < 8; ++e) zc[e] = make_float2(0.f, 0.f);
    // The rotations of the next tile's rows are asked for as soon as this tile's have been used.  Nothing may touch them
    // before their tile comes, since that waits for the load: not a copy (d = 64, where both boxes use the same: 4000 of the 5700
    // cycles that this role took a tile), and no choice between what is loaded and something else.  Rows beyond the last token
    // keep what they have (they are not stored), and the last tile asks for its own once more.
    uint4 tab0[kTileApply / 32], tab1[kTileApply / 32];
#pragma unroll
    for (int i = 0; i < kTileApply / 32; ++i) tab0[i] = tab1[i] = make_uint4(0, 0, 0, 0);
    auto fetch_rot = [&](int tile, int i) {
      const long long n = (long long)tile * kTileApply + row0 + 32 * i;
      const uint4* at = p.rope + n * (D / 8);
      load_in_place(tab0[i], at + C::tab_chunk(0, lc), n < p.N);
      if (!C::SAME_TAB) load_in_place(tab1[i], at + C::tab_chunk(1, lc), n < p.N);
    };
    if (ROPE) {
      TileWalk t0(wc);
      if (!t0.done()) {
#pragma unroll
        for (int i = 0; i < kTileApply / 32; ++i) fetch_rot(t0.tile(), i);
      }
    }
    for (TileWalk t(wc); !t.done() && ok; t.next(), ++it) {
      const int s = it % NSC;
      if (t.seg_first()) {
        // the previous segment's MMAs must be done before its S operand is overwritten
        if (seg > 0) ok = mbar_wait(seg_done, (seg - 1) & 1, abort_flag);
        if (!ok) break;
        const int u = t.unit();
        if (SOLO) {
        } else if (IMAGE) {
          if (tr == 0) {   // the unit's operand image, made by the reduce: one bulk copy
            fence_proxy_async_all();
            mbar_arrive_expect_tx(s_ready, C::S_BYTES);
            bulk_load(s_op, p.s_image + (size_t)u * C::S_BYTES, C::S_BYTES, s_ready);
          } else {
            mbar_arrive(s_ready);
          }
        } else {
          build_s_operand<D>(s_op, p.state, u / p.HG, u % p.HG, p.H, tr, R::RELU_THREADS + 128);
        }
        if (ROPE) {
          // feature 64 * box + 8 * lc of the operand is feature fl of head g of the group
#pragma unroll
          for (int box = 0; box < 2; ++box) {
            const int f0 = 64 * box + 8 * lc, g = f0 / D, fl = f0 - g * D;
            const int h = (u % p.HG) * C::G + g;
            float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
            if (SOLO) {
              if (box == 0 || box1_live) {
                a0 = *reinterpret_cast<const float4*>(z_row + f0);
                a1 = *reinterpret_cast<const float4*>(z_row + f0 + 4);
              }
            } else if ((box == 0 || box1_live) && h < p.H) {
              const float4* zrow = reinterpret_cast<const float4*>(p.state + ((size_t)((u / p.HG) * p.H + h) * (D + 1) + D) * D);
              a0 = __ldcg(zrow + fl / 4);
              a1 = __ldcg(zrow + fl / 4 + 1);
            }
            zc[4 * box + 0] = make_float2(a0.x, a0.y); zc[4 * box + 1] = make_float2(a0.z, a0.w);
            zc[4 * box + 2] = make_float2(a1.x, a1.y); zc[4 * box + 3] = make_float2(a1.z, a1.w);
          }
        }
        if (!SOLO && !IMAGE) {
          fence_proxy_async_smem();
          mbar_arrive(s_ready);
        }
        ++seg;
      }
      if (ROPE) {
        // numerator operand: rotated phi(q); denominator: plain phi(q) . z, added up over the eight lanes that
        // share a row and left in the row's zero padding (features 112..) for the epilogue
        uint8_t* sl = slots + s * SLOT;
        TileWalk tn = t;
        tn.next();
        if (!__all_sync(0xffffffffu, mbar_wait(&c_full[s], (it / NSC) & 1, abort_flag))) break;  // leave as a whole warp
        const int ahead = tn.done() ? t.tile() : tn.tile();
        rope_apply_rows<D>(sl, den_rows + s * C::G * kTileApply, row0, pc, lc, zc, tab0, tab1, [&](int i) { fetch_rot(ahead, i); });
        fence_proxy_async_smem();
        mbar_arrive(&c_ready[s]);
        continue;
      }
      if (QT) {
        // (the columns are free when the MMAs of the tile two before, which had them, are complete)
        bool here = mbar_wait(&c_full[s], (it / NSC) & 1, abort_flag);
        if (it >= 2) here = here && mbar_wait(&c_tfull[it & 1], ((it - 2) >> 1) & 1, abort_flag);
        if (!__all_sync(0xffffffffu, here)) break;   // leave as a whole warp
        const int wq = warp & 3;
        tcgen05_fence_after();
        relu_row_to_tmem<C::FEAT>(slots + s * SLOT, HALF, wq * 32 + lane, tmem_base + (it & 1) * kAccStride + QT_COL + ((uint32_t)(wq * 32) << 16));
        tcgen05_fence_before();
        mbar_arrive(&c_ready[s]);
        continue;
      }
      if (!mbar_wait(&c_full[s], (it / NSC) & 1, abort_flag)) break;
      relu_pass<C::FEAT, kTileApply>(slots + s * SLOT, slots + s * SLOT + HALF, tr);
      fence_proxy_async_smem();
      mbar_arrive(&c_ready[s]);
    }
  } else if (warp < R::STORE_WARP) {
    // ------------------------------------------------------------ epilogue: divide, round, stage the O tile
    const int wq = warp & 3;
    const int te = threadIdx.x - R::EPI_THREAD0;
    const int r = wq * 32 + lane;  // accumulator lane = token row of the tile
    uint32_t it = 0;
    for (TileWalk t(wc); !t.done(); t.next(), ++it) {
      const int s = it % NSC;
      if (!SOLO && t.seg_first()) {
        // this thread has seen the last accumulator of the previous segment complete: S may be rebuilt
        const int u = t.unit();
        if (!IMAGE) {
          build_s_operand<D>(s_op, p.state, u / p.HG, u % p.HG, p.H, R::RELU_THREADS + te, R::RELU_THREADS + 128);
          fence_proxy_async_smem();
        }
        mbar_arrive(s_ready);
      }
      const uint32_t acc = it & 1;
      bool ok = mbar_wait(&c_tfull[acc], (it >> 1) & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tcgen05_fence_after();
      if (t.seg_last()) mbar_arrive(seg_done);
      apply_epilogue<D, ROPE>(tmem_base, acc, slots, s, den_rows, wq, r, p.eps, c_tempty);
      fence_proxy_async_smem();
      mbar_arrive(&c_staged[s]);
    }
  } else {
    // ------------------------------------------------------------ store warp: O tiles out, slots back to the producer
    if (lane == 0) {
      uint32_t it = 0;
      // A head row that is not a whole number of 128-byte lines (d = 112) shares lines with its neighbours,
      // and each head's part of such a line arrives from another SM: the O tiles are stored with the L2
      // evict-last policy so that a line is still there when its other part comes, and goes to DRAM once,
      // whole (measured: 5 % on the forward; evict-first on the K, V loads helped the state pass alone but
      // not the forward, on the Q loads it brought the over-fetch of shared lines back).
      constexpr bool kKeepStores = (C::FEAT * 2) % 128 != 0;
      const uint64_t store_policy = kKeepStores ? make_l2_policy_evict_last() : 0;
      for (TileWalk t(wc); !t.done(); t.next(), ++it) {
        const int s = it % NSC;
        if (!mbar_wait(&c_staged[s], (it / NSC) & 1, abort_flag)) break;
        const int u = t.unit(), b = u / p.HG, hg = u % p.HG;
        uint8_t* sl = slots + s * SLOT;
        int c0, c1;
        box_coords<D>(0, hg, c0, c1);
        if (kKeepStores) {
          tma_store_4d_hint(&map_o, sl, c0, c1, t.tile() * kTileApply, b, store_policy);
          box_coords<D>(1, hg, c0, c1);
          tma_store_4d_hint(&map_o, sl + HALF, c0, c1, t.tile() * kTileApply, b, store_policy);
        } else {
          tma_store_4d(&map_o, sl, c0, c1, t.tile() * kTileApply, b);
          box_coords<D>(1, hg, c0, c1);
          tma_store_4d(&map_o, sl + HALF, c0, c1, t.tile() * kTileApply, b);
        }
        tma_store_commit();
        tma_store_wait_read();
        mbar_arrive(&c_empty[s]);
      }
      tma_store_wait_all();
    }
  }

  // ------------------------------------------------------------ teardown
  tcgen05_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      p.ctrl->status = LINATTN_ERR_TIMEOUT;
      // loads still in flight target this CTA's shared memory: give each stage a bounded wait
      for (int s = 0; s < NSA + NSC; ++s)
        for (int par = 0; par < 2; ++par)
          for (int spin = 0; spin < 4096 && !mbar_try_wait(s < NSA ? &a_full[s] : &c_full[s - NSA], par); ++spin)
            __nanosleep(64);
      for (int spin = 0; SOLO && p.accumulate && spin < 4096 && !mbar_try_wait(st_full, 0); ++spin) __nanosleep(64);
    }
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

#include "umma_cluster.cuh"

// ============================================================================ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return (EncodeTiledFn) nullptr;
    return (EncodeTiledFn)f;
  }();
  return fn;
}

// 4-D bf16 map over (feature, head, token, batch) with a (box_d, box_h, tokens, 1) box, 128-byte swizzle,
// zero fill outside the tensor.
bool make_map(CUtensorMap* map, const Problem& p, const void* base, int box_d, int box_h, int box_tokens) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {(cuuint64_t)p.d, (cuuint64_t)p.H, (cuuint64_t)p.N, (cuuint64_t)p.B};
  cuuint64_t strides[3] = {(cuuint64_t)p.sh * 2, (cuuint64_t)p.sn * 2, (cuuint64_t)p.sb * 2};
  if (p.d == 32) {
    // A 64-byte box row would be padded to the 128-byte swizzle pitch, so with d = 32 (heads contiguous:
    // stride_h = 32) the heads of a token are one row of H*32 features and a box takes 64 of them (two heads).
    dims[0] = (cuuint64_t)p.H * 32; dims[1] = 1;
    strides[0] = (cuuint64_t)p.sn * 2;
  }
  cuuint32_t box[4] = {(cuuint32_t)box_d, (cuuint32_t)box_h, (cuuint32_t)box_tokens, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// SM count of the current device (0: not an sm_100 device, or no cooperative launch).
int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!cached[dev]) {
    int n = 0, major = 0, coop = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess || major != 10) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    cached[dev] = n > kMaxCtas ? kMaxCtas : n;
  }
  return cached[dev];
}

// One CTA per unit instead of all CTAs on all units?  A lone CTA takes about 4 us and 2 (packed heads) to 3 us for every 64
// tokens of its unit; the grid takes 14 to 18 us (two grid barriers, the partial records, the reduce and the operand images
// between the passes; 10 to 14 without an apply pass) and a time that grows with all units' tokens together.  Measured, launches
// back to back, lone CTAs against the grid, in us:
//                       64 tokens                  128                        192                        256
//                       forward  step  state       forward  step  state       forward  step  state       forward  step  state
//   d = 112, 1 unit     7.2/16.4 7.8/16.4 6.0/12.4 10.1/14.6 10.9/16.4 8.3/10.3 13.7/14.4 14.6/14.4 11.1/10.3 16.6/14.4 17.5/14.4 13.8/10.3
//            20         7.6/17.9 8.1/18.5 5.9/14.4 10.4/16.4 11.1/18.4 8.5/12.3 14.0/16.4 14.8/16.4 11.3/11.5 16.9/16.4 17.7/16.4 14.0/11.7
//            60         8.1/18.5 8.6/18.5 6.1/14.4 10.8/17.6 11.5/18.5 8.6/12.4 14.2/18.5 15.0/18.5 11.3/12.4 17.2/18.5 17.9/18.6 14.0/12.4
//            148        10.0/20.5 10.6/20.6 6.9/14.4 12.5/22.5 13.4/22.6 9.2/14.4 15.5/22.6 16.6/22.6 11.9/14.7 18.4/24.6 19.3/24.6 14.7/16.4
//   d = 128, 18 units   7.7/18.5 8.6/18.5 6.3/15.2 10.6/16.4 11.8/18.4 8.8/12.4 14.4/16.4 15.6/16.4 11.8/12.3 17.4/16.4 18.7/16.4 14.7/11.8
//   d = 64, 35          7.9/18.5 8.5/18.5 5.9/12.3 10.2/16.8 11.0/16.5 7.8/10.9 13.0/17.9 13.8/18.2 10.0/10.3 15.5/18.5 16.3/18.5 12.2/11.2
//   d = 32, 1           7.1/14.4 7.4/14.4 5.8/10.3 9.1/14.4 9.4/14.4 6.6/10.3 11.5/14.4 11.8/14.4 8.2/10.3 13.2/14.4 13.6/14.4 9.7/9.9
// with rotary factors alike at d = 112 and 128 and twice as fast as the grid at d = 32 and 64.  (The grid's calls in a row come out at multiples of
// 2.05 us.)  So: up to 128 tokens, and up to 192
// with packed heads or many units where these are too many for clusters, which are asked for first (cluster_size).  The choice depends on the shape and the device, not on the call, so that all
// calls on one shape (forward, state and apply, step, peek, the token-sharded three) add up in the same order and give the same bits.
inline bool solo_pays(const Problem& p, int U, int sms) {
  return U <= sms && (p.N <= 128 || (p.N <= 192 && (p.d <= 64 || 3 * U >= 2 * sms)));
}

inline int groups_of(int d) { return d == 32 ? 4 : d == 64 ? 2 : 1; }

// Instantiates and launches the kernel: cooperatively when its CTAs wait for one another.
template <int D, bool ROPE, bool SOLO, bool IMAGE, bool PREFIX = false>
int launch_kernel(int grid, void** args, cudaStream_t stream) {
  using C = Cfg<D>;
  // the opt-in to more than 48 KB of dynamic shared memory is a per-device setting of the kernel
  static bool attr_set[64] = {false};
  constexpr size_t kSmem = SOLO ? C::SMEM_SOLO : ROPE ? C::SMEM_ROPE : C::SMEM;
  static_assert(SOLO || kSmem >= kSmemAlone, "CTAs that wait for one another");
  const void* kernel = (const void*)umma_fused_kernel<D, ROPE, SOLO, IMAGE, PREFIX>;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LINATTN_ERR_CUDA;
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem) != cudaSuccess) return LINATTN_ERR_CUDA;
    attr_set[dev] = true;
  }
  cudaLaunchAttribute at[1];
  if (SOLO) {
    at[0] = early_start();
  } else {   // (an early start as well: step of 4680 tokens 31.9 -> 31.7 us, prefill 139.4 -> 140.3, the others the same)
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(Roles<ROPE>::THREADS); cfg.dynamicSmemBytes = kSmem; cfg.stream = stream;
  cfg.attrs = at; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, args);
  if (e != cudaSuccess) { cudaGetLastError(); return LINATTN_ERR_CUDA; }
  count_launches(1);
  return LINATTN_OK;
}

// Clusters of c CTAs that are on the device together (0: none), or the error that kept the runtime from saying: a call must not
// take another form, with other low bits, because this once could not be asked.
template <int D, bool ROPE>
int clusters_at_once(int c) {
  using L = ClusterCfg<D, ROPE>;
  static std::atomic<int> cached[64][L::MOST + 1];   // by device; one more than the number, 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return LINATTN_ERR_CUDA; }
  int n = cached[dev][c].load(std::memory_order_relaxed) - 1;
  if (n < 0) {
    const void* kernel = (const void*)umma_cluster_kernel<D, ROPE>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM) != cudaSuccess) { cudaGetLastError(); return LINATTN_ERR_CUDA; }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)c, 1, 1};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(c); cfg.blockDim = dim3(Roles<ROPE>::THREADS); cfg.dynamicSmemBytes = L::SMEM;
    cfg.attrs = at; cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 0) { cudaGetLastError(); return LINATTN_ERR_CUDA; }
    cached[dev][c].store(n + 1, std::memory_order_relaxed);
  }
  return n;
}

// CTAs of a unit's cluster (0: no clusters; or an error): the most that the chip holds at once for all units, where what a cluster saves
// is more than the SMs it leaves out cost.  These are 28 of 148 with 20, 40 or 60 units (clusters of 6, 3 and 2: 22, 45 and
// 74 at once), so with n 64-token tiles to a CTA there is an n from which the grid is faster; with rotary factors, whose apply
// pass streams less per SM, it is larger, with many units too (the grid's reduce grows with them), and heads of 128, whose
// sums and operand leave two Q slots, lose early.  Read-only step, back to back, clusters against the grid (lone CTAs where
// they would be taken), us:
//                        192 tokens   300          600          1200         2400         4680
//   d = 112,  4 heads    10.9/16.4    11.4/16.3    11.8/16.4    13.8/16.4    16.1/16.4    21.9/18.5
//            20          11.4/16.4    13.3/16.4    13.8/16.4    16.5/18.5    19.9/22.0    27.9/28.7
//            40          12.7/16.7    13.7/18.5    16.0/20.5    19.2/24.6    27.8/31.8    47.8/48.0
//            60          13.2/18.5    15.2/20.5    17.4/22.6    23.1/28.7    38.1/43.1    63.5/63.6
//   d = 64,  35          13.4/13.7    14.0/18.5    14.9/20.5    19.0/22.6    28.0/27.6    46.8/46.7
//   d = 128, 18          13.3/16.4    15.4/16.5    16.4/17.5    19.6/18.6    25.6/22.0    38.9/28.7
//   rotary, 112,  4      13.1/18.5    13.4/18.5    14.1/20.2    16.1/24.6    18.6/26.3    25.3/30.9
//                20      13.6/18.9    15.5/18.6    15.7/20.5    18.2/22.8    22.6/26.7    32.8/37.0
//                40      15.1/20.5    15.7/20.5    17.7/24.6    21.9/28.9    33.3/40.2    58.1/58.1
//                60      15.5/20.5    17.0/22.6    19.7/26.7    27.5/34.8    46.4/51.3    76.5/76.7
//   rotary, 64,  35      14.6/16.4    14.5/20.5    16.3/22.6    20.4/26.7    31.2/34.9    55.6/55.4
//   rotary, 128, 18      14.1/20.5    16.7/20.5    16.8/20.5    19.3/24.6    25.0/27.5    37.1/36.9
// Up to 128 tokens lone CTAs are as fast or faster (steps of 20 heads of 112 11.2 against 11.8, of 18 of 128 11.9 against 14.3; states alone 8.7 and 8.3).  S is as far from 64 bits as the
// grid's or closer (4680 tokens, 20 heads: 9.0e-8 against 1.20e-7; rotary: see the kernel's MMA issuer).  The choice depends on the shape and on the device (how its SMs
// are spread over GPCs), as the grid's split depends on its SM count: all calls on one shape give the same bits on one GPU.
//
// The fewer SMs the clusters take, the earlier the grid, which takes them all, is ahead: below two thirds of them from nine 64-token
// tiles to a CTA on (heads of 112), below three quarters from thirteen.  Few units put that off, since a unit's reduce in the grid
// adds up the records of 148 / units CTAs.  Packed heads, whose grid form is slower, lose at thirteen tiles with 3 to 9 units and
// rotary factors, and at twelve without and below two thirds.  Read-only step and state alone, from CUDA graphs, clusters against the
// grid, us:
//   rotary, 112,  4 units, 12 tiles of 8 CTAs   28.3/30.3  15.6/20.0   13 tiles   30.0/31.0  16.2/20.3
//                 6        10                   25.9/28.4  14.5/18.3   11         27.5/28.7  15.1/18.8
//                 8         8                   23.8/24.4  13.9/15.8    9         25.9/24.9  14.5/16.1    13  31.1/27.9  16.9/17.5
//                12         8                   24.0/26.1  14.2/16.2    9         26.1/26.4  14.8/16.5    12  30.0/30.1  16.6/17.6
//                16         8         6 CTAs    24.2/25.7  14.3/15.7    9         26.3/26.0  14.9/15.8    13  32.5/32.2  17.3/17.8
//                18        12         6 CTAs    30.3/32.3  16.9/17.9   13         33.0/33.2  17.4/18.5
//                26        13         5 CTAs    36.0/39.2  18.8/20.0
//                33        13         4 CTAs    34.8/39.7  17.9/19.8
//                35        12         3 CTAs    30.2/31.2  16.8/17.1   13         32.8/32.3  17.5/17.8
//                46         8         2 CTAs    23.7/25.5  15.1/15.5    9         25.7/25.5  15.7/15.5    12  30.4/29.1  17.6/16.8
//                50        12         2 CTAs    31.3/37.3  17.6/20.4
//   d = 112,     46         8         2 CTAs    20.1/20.8  12.5/12.3    9         21.6/20.8  13.2/12.4    12  25.2/23.5  15.1/13.4
//   rotary, 64,   8        12         8 CTAs    27.7/27.7  13.7/17.0   13         29.5/27.8  14.2/17.2
//   d = 64,      46        11         2 CTAs    24.5/22.8  13.4/12.8   12         25.5/23.4  14.0/12.8
//   d = 32,      33         4         4 CTAs    14.9/17.6   8.0/10.2
//   rotary, 32,  22        13         6 CTAs    34.3/42.1  13.6/18.7
//   d = 128,     18         1         3 CTAs    13.0/15.2   9.7/10.6
//   rotary, 128, 18         4         6 CTAs    19.1/23.1  12.8/14.1
//                26         1         5 CTAs    17.7/18.8  12.4/11.7
// One form for all calls: states alone lose up to 9 % on clusters with 46 to 49 units from six tiles on.
// Not taken though clusters would be ahead (the line was drawn before early starts, which shorten clusters and not the grid): plain heads of 112 from
// three tiles to a CTA on in clusters of four and more (20 units 15.5/17.0 at three tiles, 26.2/27.2 at twelve, level at thirteen; 33 units 15.5/17.6 at
// three), and from thirteen on with 38 to 45 and 50 to 74 units (40 units 27.6/30.5, 60 27.5/32.2).  Taken though the grid would be: packed heads
// without rotary factors, 46 to 49 units of eleven tiles.
template <int D, bool ROPE>
int cluster_size(const Problem& p, int U, long long tiles, int sms) {
  if (p.N <= 128) return 0;
  for (int c = tiles < 8 ? (int)tiles : 8; c >= 2; --c) {
    const int at_once = clusters_at_once<D, ROPE>(c);
    if (at_once < 0) return at_once;
    if (at_once < U) continue;
    int most = ROPE ? (D == 128 ? 4 : c == 2 ? 12 : 13) : D == 128 ? (p.N <= 192 ? 1 : 0) : c <= 3 ? 12 : D == 112 ? 2 : 4;
    const int used = U * c;   // SMs
    int few = most;
    if (D == 112 && 3 * used < 2 * sms) few = U <= 2 ? 13 : U <= 4 ? 12 : U <= 6 ? 10 : 8;
    else if (D == 112 && 4 * used <= 3 * sms) few = 12;
    else if (D <= 64 && ROPE && 2 * used < sms) few = U <= 2 ? 13 : 12;
    else if (D <= 64 && !ROPE && 3 * used < 2 * sms) few = 11;
    if (few < most) most = few;
    return (tiles + c - 1) / c <= most ? c : 0;
  }
  return 0;
}

template <int D, bool ROPE>
int launch_cluster(const Problem& p, const UmmaCall& c, int size, int U, void* workspace, cudaStream_t stream) {
  using C = Cfg<D>;
  using L = ClusterCfg<D, ROPE>;
  ClusterParams cp{};
  cp.H = p.H; cp.HG = (p.H + C::G - 1) / C::G;
  cp.tiles = (int)((p.N + kTileState - 1) / kTileState);
  cp.c = size;
  cp.do_apply = c.q != nullptr; cp.accumulate = c.accumulate ? 1 : 0;
  cp.state = c.state;
  cp.state_base = c.state_base ? c.state_base : c.state;
  // in a launch that applies, only a cache that takes the block needs the sum in memory
  cp.write_state = !cp.do_apply || (c.accumulate && cp.state_base == cp.state);
  cp.eps = c.eps;
  cp.ctrl = static_cast<WorkspaceCtrl*>(workspace);
  cp.rope = static_cast<const uint4*>(c.rope);
  cp.N = p.N;
  CUtensorMap mk, mv, mq, mo;
  if (!make_map(&mk, p, c.k, C::BOX_D, C::BOX_H, kTileState) || !make_map(&mv, p, c.v, C::BOX_D, C::BOX_H, kTileState)) return LINATTN_ERR_CUDA;
  mq = mk; mo = mk;   // (never used without queries)
  if (cp.do_apply && (!make_map(&mq, p, c.q, C::BOX_D, C::BOX_H, kTileState) || !make_map(&mo, p, c.o, C::BOX_D, C::BOX_H, kTileState)))
    return LINATTN_ERR_CUDA;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)size, 1, 1};
  at[1] = early_start();
  bool early = true;
  if (size > 2 && size % 2) {
    const int at_once = clusters_at_once<D, ROPE>(size), wider = clusters_at_once<D, ROPE>(size + 1);
    if (at_once <= 0 || wider < 0) return LINATTN_ERR_CUDA;
    early = clusters_start_early(size, U, at_once, wider, (cp.tiles + size - 1) / size);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(size * U); cfg.blockDim = dim3(Roles<ROPE>::THREADS); cfg.dynamicSmemBytes = L::SMEM; cfg.stream = stream;
  cfg.attrs = at; cfg.numAttrs = early ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, umma_cluster_kernel<D, ROPE>, mk, mv, mq, mo, cp) != cudaSuccess) { cudaGetLastError(); return LINATTN_ERR_CUDA; }
  count_launches(1);
  return LINATTN_OK;
}

template <int D, bool ROPE>
int launch_fused(const Problem& p, const UmmaCall& c, void* workspace, cudaStream_t stream) {
  using C = Cfg<D>;
  const int sms = sm_count();
  if (!sms) return LINATTN_ERR_CUDA;
  const bool do_state = c.k != nullptr, do_apply = c.q != nullptr;
  FusedParams fp{};
  fp.B = p.B; fp.H = p.H; fp.HG = (p.H + C::G - 1) / C::G;
  const int U = p.B * fp.HG;
  const bool prefill = c.blocks > 1;   // (asked for where it pays, see umma_joins_prefill: always the grid)
  if (do_state && !prefill) {
    const int size = cluster_size<D, ROPE>(p, U, (p.N + kTileState - 1) / kTileState, sms);
    if (size < 0) return size;
    if (size) return launch_cluster<D, ROPE>(p, c, size, U, workspace, stream);
  }
  fp.sa = make_sched(U, (p.N + kTileState - 1) / kTileState, sms, 2);
  fp.do_state = do_state; fp.do_apply = do_apply; fp.accumulate = c.accumulate ? 1 : 0;
  fp.state = c.state;
  fp.state_base = c.state_base ? c.state_base : c.state;
  fp.partials = reinterpret_cast<float*>(static_cast<char*>(workspace) + LINATTN_WORKSPACE_CTRL_BYTES);
  fp.eps = c.eps;
  fp.ctrl = static_cast<WorkspaceCtrl*>(workspace);
  fp.rope = static_cast<const uint4*>(c.rope);
  fp.N = p.N;
  fp.s_image = nullptr;
  fp.blocks = c.blocks;
  fp.cache = c.cache;
  if (do_state && do_apply && C::G == 1 && (fp.sa.P >= 1 || prefill)) {
    // The operand images live at the end of the partials area, which is sized for kMaxCtas + U records while a
    // launch writes at most P*U + R + U of them: used when they fit behind the records in use.
    const size_t rec_bytes = ((size_t)p.state_elems() + (ROPE ? kZParts : 0)) * sizeof(float);
    const size_t used = ((size_t)fp.sa.P * U + fp.sa.R + U) * rec_bytes;
    const size_t img = (size_t)U * C::S_BYTES;
    size_t total = umma_partial_bytes(p, ROPE);
    if (prefill) total = (size_t)(reinterpret_cast<char*>(c.state) - reinterpret_cast<char*>(fp.partials)) + (size_t)U * p.state_elems() * sizeof(float);   // (the images take the place of the states)
    if (total >= img + 1024) {
      const size_t off = (total - img) & ~(size_t)1023;
      if (off >= used) fp.s_image = reinterpret_cast<uint8_t*>(fp.partials) + off;
    }
  }
  // a unit switch costs the apply pass about one tile when the S operand comes as an image, two when the CTA
  // builds it from the fp32 state
  fp.sc = make_sched(U, (p.N + kTileApply - 1) / kTileApply, sms, fp.s_image ? 1 : 2);
  const bool solo = do_state && !prefill && solo_pays(p, U, sms);
  if (solo) {
    fp.sa.U = fp.sc.U = fp.sa.grid = fp.sc.grid = U;
    fp.sa.P = fp.sc.P = 1;
    fp.sa.R = fp.sc.R = fp.sa.m = fp.sc.m = 0;
    fp.sa.Lc = fp.sa.tpu;
    fp.sc.Lc = fp.sc.tpu;
    // in a launch that applies, only a cache that takes the block needs the sum in memory
    fp.write_state = !do_apply || (c.accumulate && fp.state_base == fp.state);
  }
  int grid = 0;
  if (do_state) grid = fp.sa.grid;
  if (do_apply && fp.sc.grid > grid) grid = fp.sc.grid;
  CUtensorMap mk, mv, mq, mo;
  if (do_state) {
    if (!make_map(&mk, p, c.k, C::BOX_D, C::BOX_H, kTileState) || !make_map(&mv, p, c.v, C::BOX_D, C::BOX_H, kTileState))
      return LINATTN_ERR_CUDA;
  }
  if (do_apply) {
    if (!make_map(&mq, p, c.q, C::BOX_D, C::BOX_H, kTileApply) || !make_map(&mo, p, c.o, C::BOX_D, C::BOX_H, kTileApply))
      return LINATTN_ERR_CUDA;
  } else {
    mq = mk; mo = mk;  // never dereferenced
  }
  if (!do_state) { mk = mq; mv = mq; }
  void* args[] = {&mk, &mv, &mq, &mo, &fp};
  if constexpr (!ROPE) {
    if (prefill) return C::G == 1 && fp.s_image ? launch_kernel<D, false, false, C::G == 1, true>(grid, args, stream) : launch_kernel<D, false, false, false, true>(grid, args, stream);
  }
  if (solo) return launch_kernel<D, ROPE, true, false>(grid, args, stream);
  if (C::G == 1 && fp.s_image) return launch_kernel<D, ROPE, false, C::G == 1>(grid, args, stream);
  return launch_kernel<D, ROPE, false, false>(grid, args, stream);
}

}  // namespace

bool umma_supported(const Problem& p) {
  // d = 32 packs four heads into one operand row, which needs the heads of a token to be contiguous
  return p.dtype == LINATTN_BF16 && (p.d == 64 || p.d == 112 || p.d == 128 || (p.d == 32 && p.sh == 32)) &&
         p.N < (1ll << 31) && p.sh * 2 < (1ll << 40) && p.sn * 2 < (1ll << 40) && p.sb * 2 < (1ll << 40);
}

// One partial record (G head-states) per (CTA, unit) segment of the state pass: at most kMaxCtas + units.
size_t umma_partial_bytes(const Problem& p, bool rope) {
  const int G = groups_of(p.d);
  const size_t units = (size_t)p.B * ((p.H + G - 1) / G);
  return ((size_t)kMaxCtas + units) * (G * (size_t)p.state_elems() + (rope ? kZParts : 0)) * sizeof(float);
}

// The rotary variant runs on the tensor cores wherever the plain kernel does.  d = 112, the paper's: the denominators
// travel in the zero padding of the 112-feature rows; every other head dim: in a small shared-memory array per slot
// and head of the group.  With packed heads (d = 32, 64) both boxes of a row use the same 16-byte chunk of the
// rotation table, since box 1 starts a new head.  Everything else takes the fp32-accurate kernels.
bool umma_rope_supported(const Problem& p) { return umma_supported(p); }

template <int D, bool ROPE>
int cluster_ctas(const Problem& p) {
  const int sms = sm_count();
  if (!sms) return LINATTN_ERR_CUDA;
  return cluster_size<D, ROPE>(p, p.B * ((p.H + Cfg<D>::G - 1) / Cfg<D>::G), (p.N + kTileState - 1) / kTileState, sms);
}

// One launch for all blocks, or a state launch, prefix_states and an apply launch?
//
// One launch where the grid takes the blocks' state anyway.  Lone CTAs and clusters keep their chains of the tensor core's additions at one and two, in
// the grid they are as long as a CTA has tiles: blocks that the former take would get sums further from 64 bits, and others than the
// same call without queries gives.  S, relative, one launch / three: 2 blocks of 2304 tokens, 20 heads of 112 1.20e-7 / 8.8e-8, 4 of 900, 35 heads of 64
// 1.10e-7 / 8.0e-8, 7 of 128, 70 heads of 32 7.1e-8 / 6.8e-8; never the other way round.  (One launch would be the faster one there: 18.6 / 28.8 us
// for 7 blocks of 64 tokens, 20 heads of 112.)
//
// And not for few heads: a thread of reduce_prefix walks the records of all blocks of its piece, CTAs / head groups of them, eight at a
// time: 49 with three groups, 74 with two, 148 with one.  The line is at 64 for every head dim and any number of blocks.  At 74 heads of 112 and
// 128 would still gain a little, packed heads lose, at 148 all lose.  One launch / three, us (-: lone CTAs or clusters take the blocks):
//                       tokens a block    300        600        1200       2400       4680
//   d = 112, 20 groups, 7 blocks          22.6/34.9  28.7/40.2  45.2/59.8  68.6/84.2  122/138
//             3         7                 -          -          25.8/28.6  28.8/32.8  37.0/40.5
//             2         7                 -          -          26.7/28.1  28.8/28.3  33.2/34.1
//             2         2                 -          -          20.6/24.7  22.6/24.7  27.4/28.8   (38, 74, 74 records)
//             1         7                 -          -          34.9/26.7  36.5/27.3  38.4/29.5
//   d = 64,   2         7                 -          -          -          30.8/28.5  34.9/34.9
//   d = 32,   2         7                 -          -          -          28.8/26.7  34.3/32.9
//   d = 128, 20         7                 22.6/39.0  32.9/49.3  49.4/65.9  76.7/94.5
//             2         7                 20.6/27.7  26.7/28.7  27.4/28.5  29.0/31.9  34.5/36.8   (35, 70, 74, 74, 74)
//             1         7                 20.6/26.6  26.7/28.0  36.7/28.1  36.9/27.7  39.0/32.1   (35, 70, 133, 148, 148)
template <int D>
bool joins_prefill(const Problem& p, int blocks) {
  const int sms = sm_count(), hg = (p.H + Cfg<D>::G - 1) / Cfg<D>::G;
  if (!sms || cluster_ctas<D, false>(p) || solo_pays(p, p.B * hg, sms)) return false;   // (an error here is the state launch's to report)
  const long long groups = (long long)(p.B / blocks) * hg, tiles = groups * blocks * ((p.N + kTileState - 1) / kTileState);
  return (tiles < sms ? tiles : sms) <= 64 * groups;
}

bool umma_joins_prefill(const Problem& p, int blocks) {
  switch (p.d) {
    case 32: return joins_prefill<32>(p, blocks);
    case 64: return joins_prefill<64>(p, blocks);
    case 112: return joins_prefill<112>(p, blocks);
    case 128: return joins_prefill<128>(p, blocks);
  }
  return false;
}

int umma_cluster_ctas(const Problem& p, bool rope) {
  switch (p.d) {
    case 32: return rope ? cluster_ctas<32, true>(p) : cluster_ctas<32, false>(p);
    case 64: return rope ? cluster_ctas<64, true>(p) : cluster_ctas<64, false>(p);
    case 112: return rope ? cluster_ctas<112, true>(p) : cluster_ctas<112, false>(p);
    case 128: return rope ? cluster_ctas<128, true>(p) : cluster_ctas<128, false>(p);
  }
  return 0;
}

int umma_run(const Problem& p, const UmmaCall& c, void* workspace, cudaStream_t stream) {
  if (p.N == 0 || (!c.k && !c.q)) return LINATTN_OK;
  switch (p.d) {
    case 32: return c.rope ? launch_fused<32, true>(p, c, workspace, stream) : launch_fused<32, false>(p, c, workspace, stream);
    case 64: return c.rope ? launch_fused<64, true>(p, c, workspace, stream) : launch_fused<64, false>(p, c, workspace, stream);
    case 112: return c.rope ? launch_fused<112, true>(p, c, workspace, stream) : launch_fused<112, false>(p, c, workspace, stream);
    case 128: return c.rope ? launch_fused<128, true>(p, c, workspace, stream) : launch_fused<128, false>(p, c, workspace, stream);
  }
  return LINATTN_ERR_UNSUPPORTED;
}

}  // namespace linattn
