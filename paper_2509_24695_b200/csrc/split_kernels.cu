// fp32-accurate state and apply passes on the tensor cores: fp32 tensors, and the bf16 head dims the fused kernel
// (umma_kernels.cu) does not take, wherever rows can be read in 16-byte pieces (split_ok).
//
// An fp32 value is the sum of three bf16 values exactly: 8 significand bits each, rounded to nearest, so that a value in
// [2^a, 2^(a+1)) leaves at most 2^(a-8) to the second part and 2^(a-16) to the third, of either sign.  A product of two such
// sums is nine bf16 products, exact in the tensor core's fp32 accumulators.  Six are taken.  Of the other three two are up
// to 2^-24 of the product of the leading powers of two each (2^-26 on average, without bias; a multiply-add rounds to 2^-24)
// and one is below 2^-31; inputs of one tile, where nothing averages out, have the two as well.  (Parts cut off instead of
// rounded all have the value's sign: then the two reach 2^-21 and add up.  All inputs with eight products: 480p layer,
// state 173 -> 190 us, apply 183 -> 217.)  What is left to chance is how the products are added up.  The tensor core
// truncates when it adds into an accumulator (2^-24 on average, always towards zero), so (1) the leading products have
// accumulators apart from the small ones, whose additions are 2^-8 below; (2) they are dealt over several accumulators, so
// that no chain is longer than two or three; and (3) the accumulators are added up in registers, round to nearest, every 32
// to 128 tokens.  bf16 operands are one part, rotated ones three; S is always three.  z and the denominators are plain fp32
// sums.  Distance from 64 bits (2-norm, S / outputs), against the general kernels' chains of fp32 multiply-adds: normal data
// 1.0 / 0.5 times theirs at one token, 0.65 / 0.5 at 8, 0.4 / 0.5 at 64 and 0.2 to 0.3 / 0.4 from 512 on; one-sign and
// log-normal data 1.0 at one token and less than theirs beyond.
//
// Parts end where bf16 does: a value below 2^-110 loses up to 2^-134, an infinity or a value above 3.396e38 has no parts
// (Inf - Inf), and products of parts end at 2^-149.  So a CTA whose sums are not finite, or so small beside its data that this would show, does its
// share again by plain fp32 multiply-adds, from memory (state_by_fma, apply_by_fma): the result is theirs, infinities and
// NaN included.  The bounds are far from what data of one scale give: they are looked at once per CTA or token row.
//
// Operand layouts are those of the fused kernel: 128-byte swizzled rows of 64 features.  Every thread reads its own
// pieces with private asynchronous copies, rectifies, rotates and splits them, and stores the parts; one thread issues
// the MMAs, and other warps drain the accumulators.  Waits on barriers are on this CTA's own work and bounded.  Two are not:
// the CTAs of a cluster meet (cluster_sync; each gets there, since its other waits are bounded), and tensor memory is
// allocated before it (no other CTA can hold it for good: kSmemAlone).
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace linattn {
namespace {

using namespace ptx;

// Warp roles: 0..7 prepare tiles (load, rectify, rotate, split), 8..15 drain accumulators (and store), 16 issues the MMAs.
// The roles only meet at barriers, two tiles apart at most; with all sixteen warps doing both in turn a tile took the sum
// of the two instead of the longer one.
constexpr int kPrepare = 256;
constexpr int kDrain = 256;
constexpr int kMmaWarp = (kPrepare + kDrain) / 32;
constexpr int kBlock = kPrepare + kDrain + 32;
// Barriers and flags of a CTA.  (The raw pieces follow: 80 bytes in their place cost bf16 heads of 96 14 % of the apply pass.)
constexpr int kBarBytes = 128;

template <typename T>
struct Piece;   // 16 bytes of a row
template <>
struct Piece<float> {
  static constexpr int E = 4;
  using Tab = uint2;   // the (cos, sin) fp16 pairs of its feature pairs
};
template <>
struct Piece<__nv_bfloat16> {
  static constexpr int E = 8;
  using Tab = uint4;
};

// What both passes know about a shape.  R = ceil(d / 16).
template <typename T, int R, bool ROPE>
struct Shape {
  static constexpr int E = Piece<T>::E;
  static constexpr int DP = 16 * R;                        // features with padding
  static constexpr int BOXES = (DP + 63) / 64;
  static constexpr bool F32 = sizeof(T) == 4;
  static constexpr int QK_PARTS = F32 || ROPE ? 3 : 1;     // bf16 parts of phi(k), phi(q)
  static constexpr int V_PARTS = F32 ? 3 : 1;
  using Tab = typename Piece<T>::Tab;
};

// With `lanes` threads to a row, which bit of the piece index odd rows flip, so that the stores of the neighbouring rows of
// one shared-memory access fall into different banks (8-byte stores of fp32 pieces, 16-byte stores of bf16 ones).
__host__ __device__ constexpr int flip_of(int E, int lanes, int pieces) {
  return E == 4 ? (lanes == 8 && pieces % 2 == 0 ? 1 : lanes == 4 && pieces % 4 == 0 ? 2 : 0) : (lanes == 4 && pieces % 2 == 0 ? 1 : 0);
}

template <int BYTES>
__device__ __forceinline__ void copy_async(void* smem_dst, const void* src, bool live) {   // not live: zeros
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(live ? 8 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void widen(const uint4& r, float (&x)[4]) {
  x[0] = __uint_as_float(r.x); x[1] = __uint_as_float(r.y); x[2] = __uint_as_float(r.z); x[3] = __uint_as_float(r.w);
}
__device__ __forceinline__ void widen(const uint4& r, float (&x)[8]) {
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { x[2 * i] = __uint_as_float(w[i] << 16); x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
}

// (a, b) -> (a c - b s, b c + a s) for every feature pair of the piece
template <int E>
__device__ __forceinline__ void rotate(float (&x)[E], const __half2* tab) {
#pragma unroll
  for (int e = 0; e < E; e += 2) {
    const float2 cs = __half22float2(tab[e / 2]);
    const float a = x[e], b = x[e + 1];
    x[e] = a * cs.x - b * cs.y;
    x[e + 1] = b * cs.x + a * cs.y;
  }
}

// Byte offset of feature f (a multiple of 4) of row `row` in an operand of boxes of 64 features, `box_bytes` each.
__device__ __forceinline__ int operand_offset(int row, int f, int box_bytes) {
  return (f >> 6) * box_bytes + row * 128 + ((((f & 63) >> 3) ^ (row & 7)) << 4) + ((f & 4) << 1);
}

// The next bf16 part of every value, rounded to nearest; x becomes what is left.  Packed in pairs.
template <int E>
__device__ __forceinline__ void take_part(float (&x)[E], uint32_t (&w)[E / 2]) {
#pragma unroll
  for (int e = 0; e < E; e += 2) {
    w[e / 2] = pack_bf16x2(x[e], x[e + 1]);
    x[e] -= __uint_as_float(w[e / 2] << 16);
    x[e + 1] -= __uint_as_float(w[e / 2] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ void store_words(uint8_t* at, const uint32_t (&w)[2]) { *reinterpret_cast<uint2*>(at) = make_uint2(w[0], w[1]); }
__device__ __forceinline__ void store_words(uint8_t* at, const uint32_t (&w)[4]) { *reinterpret_cast<uint4*>(at) = make_uint4(w[0], w[1], w[2], w[3]); }

// left: collects what the last of three parts is taken from; bits in its lower half are lost.
template <int PARTS, int E>
__device__ __forceinline__ void store_parts(uint8_t* at, int part_bytes, float (&x)[E], uint32_t& left) {
#pragma unroll
  for (int s = 0; s < PARTS; ++s) {
    if (s == 2) {
#pragma unroll
      for (int e = 0; e < E; e += 2) left |= __float_as_uint(x[e]) | __float_as_uint(x[e + 1]);
    }
    uint32_t w[E / 2];
    take_part(x, w);
    store_words(at + s * part_bytes, w);
  }
}

__device__ __forceinline__ void tmem_ld_x8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

// After a wait that ran out: the MMAs that were issued still read this CTA's shared memory and write its tensor memory.
// They get a bounded time to finish before either is used for something else (whole CTA).
__device__ __forceinline__ void let_finish(uint64_t* finished) {
  if (threadIdx.x == 0)
    for (int spin = 0; spin < 4096 && !mbar_try_wait(finished, 0); ++spin) __nanosleep(64);
  __syncthreads();
}

// ---------------------------------------------------------------- by plain multiply-adds (whole CTA)
__device__ __forceinline__ void store_value(float* o, float x) { *o = x; }
__device__ __forceinline__ void store_value(__nv_bfloat16* o, float x) { *o = __float2bfloat16_rn(x); }

// Feature e of token n, rectified, as the general kernels read it: plain, and with ROPE turned.
template <typename T, bool ROPE>
__device__ __forceinline__ void phi_of(const T* row, const __half2* tab, int d, long long n, int e, float& plain, float& turned) {
  plain = turned = fmaxf((float)row[e], 0.f);
  if (ROPE) {
    const float other = fmaxf((float)row[e ^ 1], 0.f);
    const float2 cs = __half22float2(tab[n * (d / 2) + e / 2]);
    turned = (e & 1) ? other * cs.y + plain * cs.x : plain * cs.x - other * cs.y;
  }
}

// S of tokens [n0, n1) of the unit at k, v: out[j * d + i] = sum of phi(k)_i v_j, token after token.  scratch: 16 KB of shared
// memory.  32 x 16 threads with a tile of 4 x 8 sums each.
template <typename T, bool ROPE>
__device__ __noinline__ void state_by_fma(const T* k, const T* v, const __half2* tab, int d, long long sn, long long n0, long long n1,
                                          float* scratch, float* out) {
  constexpr int TOK = 16;
  float* ks = scratch;
  float* vs = scratch + TOK * 128;
  const int tid = (int)threadIdx.x, ti = tid >> 4, tj = tid & 15;
  float acc[4][8];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 8; ++s) acc[r][s] = 0.f;
  for (long long n = n0; n < n1; n += TOK) {
    __syncthreads();
    for (int idx = tid; idx < TOK * 128; idx += kBlock) {
      const int t = idx >> 7, e = idx & 127;
      float plain = 0.f, x = 0.f, y = 0.f;
      if (n + t < n1 && e < d) {
        phi_of<T, ROPE>(k + (n + t) * sn, tab, d, n + t, e, plain, x);
        y = (float)v[(n + t) * sn + e];
      }
      ks[idx] = x;
      vs[idx] = y;
    }
    __syncthreads();
    const int live = (int)min((long long)TOK, n1 - n);
    for (int t = 0; t < live && ti < 32; ++t) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float a = ks[t * 128 + ti + 32 * r];
#pragma unroll
        for (int s = 0; s < 8; ++s) acc[r][s] = fmaf(a, vs[t * 128 + tj + 16 * s], acc[r][s]);
      }
    }
  }
  __syncthreads();   // out may be where the scratch is
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int i = ti + 32 * r, j = tj + 16 * s;
      if (ti < 32 && i < d && j < d) out[j * d + i] = acc[r][s];
    }
}

// Outputs of tokens [n0, n1) of the unit at q, o against the state W.  scratch: (d * d + d + 256 * warps) floats of shared
// memory.  A warp takes a token.
template <typename T, bool ROPE>
__device__ __noinline__ void apply_by_fma(const T* q, const float* W, T* o, const __half2* tab, int d, long long sn, long long n0,
                                          long long n1, float eps, float* scratch) {
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* ss = scratch;              // S[i][j]
  float* zs = ss + d * d;           // z
  float* qs = zs + d + 256 * warp;  // this token's phi(q), turned, then plain
  float* qp = qs + 128;
  for (int idx = tid; idx < d * d; idx += kBlock) ss[(idx % d) * d + idx / d] = W[idx];
  for (int i = tid; i < d; i += kBlock) zs[i] = W[(long long)d * d + i];
  __syncthreads();
  for (long long n = n0 + warp; n < n1; n += kBlock / 32) {
    for (int e = lane; e < d; e += 32) phi_of<T, ROPE>(q + n * sn, tab, d, n, e, qp[e], qs[e]);
    __syncwarp();
    float num[4] = {0.f, 0.f, 0.f, 0.f}, den = 0.f;
    for (int i = 0; i < d; ++i) {
      den = fmaf(qp[i], zs[i], den);
#pragma unroll
      for (int s = 0; s < 4; ++s)
        if (lane + 32 * s < d) num[s] = fmaf(qs[i], ss[i * d + lane + 32 * s], num[s]);
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (lane + 32 * s < d) store_value(o + n * sn + lane + 32 * s, num[s] / (den + eps));
    __syncwarp();
  }
}

// ---------------------------------------------------------------- state
template <typename T, int R, bool ROPE>
struct StateShape : Shape<T, R, ROPE> {
  using B = Shape<T, R, ROPE>;
  // tokens of a tile: 64 where two stages of parts and three of raw pieces fit, else 32
  static constexpr int BYTES_64 = 2 * (B::QK_PARTS + B::V_PARTS) * B::BOXES * 8192 + 3 * 64 * B::DP * (2 * (int)sizeof(T) + (ROPE ? 2 : 0));
  static constexpr int TOK = BYTES_64 <= 200 * 1024 ? 64 : 32;
  static constexpr int LANES = kPrepare / TOK;               // threads to a row
  static constexpr int PIECES = (B::DP / B::E + LANES - 1) / LANES;   // 16-byte pieces of a row per thread
  static constexpr int FLIP = flip_of(B::E, LANES, PIECES);
  static constexpr int BOX = TOK * 128;
  static constexpr int PART = B::BOXES * BOX;
  static constexpr int STAGE = (B::QK_PARTS + B::V_PARTS) * PART;
  static constexpr int RAW_STAGES = 3;
  static constexpr int TAB = ROPE ? PIECES * kPrepare * (int)sizeof(typename B::Tab) : 0;
  static constexpr int RAW = 2 * PIECES * kPrepare * 16 + TAB;
  static constexpr int Z_BYTES = TOK * B::DP * 4 + 1024;      // (and the smallest sums)
  static constexpr int OWN_BYTES = (B::DP + 1) * B::DP * 4;   // a CTA's state, where its cluster reads it
  static constexpr int Z_OFF = OWN_BYTES > 2 * STAGE ? OWN_BYTES : 2 * STAGE;
  static constexpr int TAIL = Z_OFF + Z_BYTES - 2 * STAGE;
  static constexpr int NEED = 1024 + 2 * STAGE + (RAW_STAGES * RAW > TAIL ? RAW_STAGES * RAW : TAIL) + kBarBytes;
  static constexpr int SMEM = NEED > kSmemAlone ? NEED : kSmemAlone;   // (barriers last)
  static constexpr int LEAD = TOK / 32;                      // accumulators of the leading products: chains of two K steps
  static constexpr bool REST = B::QK_PARTS + B::V_PARTS > 2;
  static constexpr int ACC = B::DP <= 64 ? 64 : 128;         // TMEM columns between accumulators
  static constexpr int SET = (LEAD + (REST ? 1 : 0)) * ACC;  // one set collects a tile while the other is drained
  static constexpr int COLS = 2 * SET <= 128 ? 128 : 2 * SET <= 256 ? 256 : 512;
  static_assert(2 * SET <= 512, "tensor memory");
  static_assert(!REST || SMEM - 1024 - kBarBytes - Z_OFF >= 16384, "scratch of state_by_fma");
};

// grid (P, units): state of the tiles [c * tiles / P, (c + 1) * tiles / P) of one unit, in the library's layout.  Either
// every CTA writes a partial state (state null), or the P CTAs of a unit are a cluster and add theirs up, in the order of
// fma_state_reduce and in 64 bits as there, through distributed shared memory: state = (base ? base : 0) + sum.  No second
// kernel then, and no partial states, so that P is not bound by their room; but a cluster has to fit into one GPC (8 CTAs
// of this size at most, and 15 such clusters on the chip), so that large inputs want the other form (launch_state).
//
// Measured (32 760 tokens, 20 heads of 112, fp32; floor: 587 MB, 90 us at the copy rate): 177 us with the reduce of the
// partial states (192 with every warp preparing and draining in turn), where the general kernels take 1050 (fp32 pipe at a
// quarter of its rate, scalar loads) and a register-blocked form of them on packed fp32 FMAs 492.  A tile of 32 tokens takes
// 1.1 us, with 190 KB through shared memory (pieces in and out, their parts, 90 KB of MMA operands): two thirds of what it
// moves in that time.  (Distance from 64 bits: see the top.)
template <typename T, int R, bool ROPE>
__global__ void __launch_bounds__(kBlock, 1)
split_state_kernel(const T* __restrict__ k, const T* __restrict__ v, Problem p, int P, float* __restrict__ partials,
                   const float* base_state, float* state, const __half2* __restrict__ tab, WorkspaceCtrl* ctrl) {
  using S = StateShape<T, R, ROPE>;
  using Tab = typename S::Tab;
  constexpr int E = S::E, PIECES = S::PIECES;
  constexpr uint32_t IDESC = make_idesc_bf16(128, S::DP, true, true);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* raw = smem + 2 * S::STAGE;
  uint64_t* done = reinterpret_cast<uint64_t*>(raw + (S::SMEM - 1024 - 2 * S::STAGE - kBarBytes));   // [2] the tile's MMAs are complete
  uint64_t* ready = done + 2;                                                               // [2] the tile's parts are in its stage
  uint64_t* drained = ready + 2;                                                            // [2] its accumulators are read
  uint64_t* finished = drained + 2;                                                         // every MMA issued is complete
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(finished + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  volatile int* odd_flag = abort_flag + 1;   // the parts are not the values
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = p.d, u = blockIdx.y, c = blockIdx.x;
  const long long all = (p.N + S::TOK - 1) / S::TOK;
  const long long first = c * all / P;
  const int tiles = (int)((c + 1) * all / P - first);

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&done[i], 1); mbar_init(&ready[i], kPrepare); mbar_init(&drained[i], kDrain); }
    mbar_init(finished, 1);
    *abort_flag = *odd_flag = 0;
    fence_mbar_init();
  }
  // padded features are never written and must read as zero
  for (int i = tid; i < 2 * S::STAGE / 16; i += kBlock) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
  wait_for_prior_grids();
  if (warp == 0) { tmem_alloc(tmem_holder, S::COLS); tmem_relinquish(); }

  // preparing: this thread's row of every tile, and its pieces of it, features feature(0), feature(1), ...
  const int row = (tid % kPrepare) / S::LANES, l = tid % S::LANES;
  auto feature = [&](int i) { return (l + S::LANES * (i ^ (S::FLIP * (row & 1)))) * E; };
  const long long base = (long long)(u / p.H) * p.sb + (long long)(u % p.H) * p.sh;
  auto raw_k = [&](int st, int i) { return reinterpret_cast<uint4*>(raw + st * S::RAW) + 2 * i * kPrepare + tid; };
  auto raw_tab = [&](int st, int i) {
    return reinterpret_cast<Tab*>(raw + st * S::RAW + 2 * PIECES * kPrepare * 16) + i * kPrepare + tid;
  };
  auto issue = [&](int t, int st) {
    if (t < tiles) {
      const long long n = (first + t) * S::TOK + row;
      const bool live = n < p.N;
      const long long off = base + (live ? n : 0) * p.sn;
#pragma unroll
      for (int i = 0; i < PIECES; ++i) {
        const int f = feature(i);
        if (f >= d) continue;
        copy_async<16>(raw_k(st, i), k + off + f, live);
        copy_async<16>(raw_k(st, i) + kPrepare, v + off + f, live);
        if (ROPE) copy_async<(int)sizeof(Tab)>(raw_tab(st, i), tab + (live ? n : 0) * (d / 2) + f / 2, live);
      }
    }
    copy_commit();   // one group per tile, empty or not
  };
  float z[PIECES][E];
#pragma unroll
  for (int i = 0; i < PIECES; ++i)
#pragma unroll
    for (int e = 0; e < E; ++e) z[i][e] = 0.f;
  uint32_t left = 0;   // (a column of V so small that its sums are zero)
  auto convert = [&](int st, uint8_t* stage) {
    uint4 kr[PIECES], vr[PIECES];   // all reads before the first store: they overlap
    Tab tb[PIECES];
#pragma unroll
    for (int i = 0; i < PIECES; ++i) {
      kr[i] = *raw_k(st, i);
      vr[i] = *(raw_k(st, i) + kPrepare);
      if (ROPE) tb[i] = *raw_tab(st, i);
    }
#pragma unroll
    for (int i = 0; i < PIECES; ++i) {
      const int f = feature(i);
      if (f >= d) continue;
      float x[E];
      widen(kr[i], x);
#pragma unroll
      for (int e = 0; e < E; ++e) { x[e] = fmaxf(x[e], 0.f); z[i][e] += x[e]; }   // phi = ReLU on the keys; z from the plain ones
      if (ROPE) rotate<E>(x, reinterpret_cast<const __half2*>(&tb[i]));
      uint8_t* at = stage + operand_offset(row, f, S::BOX);
      uint32_t unused = 0;
      store_parts<S::QK_PARTS>(at, S::PART, x, unused);
      at += S::QK_PARTS * S::PART;
      if (S::V_PARTS == 1) {
        *reinterpret_cast<uint4*>(at) = vr[i];
      } else {
        widen(vr[i], x);
        store_parts<S::V_PARTS>(at, S::PART, x, left);
      }
    }
  };

  const bool preparing = tid < kPrepare;
  if (preparing) {
    issue(0, 0);
    issue(1, 1);
  }
  fence_proxy_async_smem();   // the zeros
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  let_next_grid_start();
  const uint32_t tmem = *tmem_holder;

  // draining: accumulator lane = key feature; each of the two warps of a lane quarter takes half of the value features
  constexpr int COLS = S::DP / 2;
  const int key = (warp & 3) * 32 + lane;
  const int col0 = ((warp >> 2) & 1) * COLS;
  float sum[COLS];
#pragma unroll
  for (int x = 0; x < COLS; ++x) sum[x] = 0.f;

  if (preparing) {
    for (int t = 0; t < tiles; ++t) {
      issue(t + 2, (t + 2) % S::RAW_STAGES);
      copy_wait<2>();
      if (t >= 2 && !mbar_wait(&done[t & 1], ((t - 2) >> 1) & 1, abort_flag)) break;   // the MMAs that read this stage
      convert(t % S::RAW_STAGES, smem + (t & 1) * S::STAGE);
      fence_proxy_async_smem();
      mbar_arrive(&ready[t & 1]);
    }
    copy_wait<0>();
    if (left & 0xFFFFu) *odd_flag = 1;
  } else if (warp < kMmaWarp) {
    const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16) + col0;
    for (int t = 0; t < tiles; ++t) {
      if (!__all_sync(0xffffffffu, mbar_wait(&done[t & 1], (t >> 1) & 1, abort_flag))) break;   // tcgen05.ld wants whole warps
      tcgen05_fence_after();
      if ((warp & 3) * 32 < d) {
#pragma unroll
        for (int g = 0; g < R; ++g) {
          uint32_t a[S::LEAD + 1][8];
#pragma unroll
          for (int s = 0; s < S::LEAD + (S::REST ? 1 : 0); ++s) tmem_ld_x8(trow + (t & 1) * S::SET + s * S::ACC + 8 * g, a[s]);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            float add = __uint_as_float(a[0][x]);
            if (S::LEAD > 1) add += __uint_as_float(a[S::LEAD > 1 ? 1 : 0][x]);
            if (S::REST) add += __uint_as_float(a[S::LEAD][x]);
            sum[8 * g + x] += add;
          }
        }
      }
      tcgen05_fence_before();
      mbar_arrive(&drained[t & 1]);
    }
  } else if (lane == 0) {
    int t = 0;
    for (; t < tiles; ++t) {
      if (t >= 2 && !mbar_wait(&drained[t & 1], ((t - 2) >> 1) & 1, abort_flag)) break;
      if (!mbar_wait(&ready[t & 1], (t >> 1) & 1, abort_flag)) break;
      tcgen05_fence_after();
      constexpr uint32_t LBO = S::BOXES > 1 ? S::BOX : 0;   // 64 features: rows 64..127 of the MMA repeat them and are ignored
      // shared-memory addresses are below 2^18, so an offset of a multiple of 16 bytes is added to a descriptor as it is
      const uint64_t a0 = make_smem_desc_sw128(smem_u32(smem + (t & 1) * S::STAGE), LBO, 1024), b0 = a0 + S::QK_PARTS * S::PART / 16;
      const uint32_t set = tmem + (t & 1) * S::SET;
      auto mma = [&](int kk, int pk, int pv, uint32_t acc, bool add) {
        umma_bf16(set + acc * S::ACC, a0 + (pk * S::PART + kk * 2048) / 16, b0 + (pv * S::PART + kk * 2048) / 16, IDESC, add ? 1u : 0u);
      };
      if (S::REST) {   // smallest first
        bool add = false;
#pragma unroll
        for (int order = 3; order >= 1; --order)
#pragma unroll
          for (int pk = order; pk >= 0; --pk) {
            const int pv = order - pk;
            if (pk >= S::QK_PARTS || pv >= S::V_PARTS || (order == 3 && p.N > S::TOK)) continue;
#pragma unroll
            for (int kk = 0; kk < S::TOK / 16; ++kk) { mma(kk, pk, pv, S::LEAD, add); add = true; }
          }
      }
#pragma unroll
      for (int kk = 0; kk < S::TOK / 16; ++kk) mma(kk, 0, 0, kk % S::LEAD, kk >= S::LEAD);
      umma_commit(&done[t & 1]);
    }
    if (t > 0) umma_commit(finished); else mbar_arrive(finished);
  }
  __syncthreads();
  const bool aborted = *abort_flag != 0;
  if (aborted) let_finish(finished);

  // W[j][i] = S[i][j], W[d][i] = z[i]; z's rows are added up in the raw pieces' room, behind what a cluster's state takes
  float* own = reinterpret_cast<float*>(smem);
  if (!aborted) {
    float* out = state ? own : partials + ((long long)u * P + c) * p.state_elems();
    float* zs = reinterpret_cast<float*>(smem + S::Z_OFF);   // [row][d]
    float* least = zs + S::TOK * S::DP;                      // [2][128] smallest sum of a key feature, by half of the columns
    if (!preparing && warp < kMmaWarp && key < d) {
      uint32_t low = 0xFFFFFFFFu;   // twice the bits less one: zero is the largest
      float rest = 0.f;             // NaN if a sum is not finite
#pragma unroll
      for (int x = 0; x < COLS; ++x) {
        if (col0 + x >= d) continue;
        out[(col0 + x) * d + key] = sum[x];
        if (S::REST) {
          low = min(low, 2 * __float_as_uint(sum[x]) - 1);
          rest = fmaf(sum[x], 0.f, rest);
        }
      }
      if (S::REST)   // (a sum that is not finite: 0; nothing but zeros: the largest number)
        least[(warp >> 2 & 1) * 128 + key] = rest != 0.f ? 0.f : __uint_as_float(low == 0xFFFFFFFFu ? 0x7F7FFFFFu : (low >> 1) + 1);
    }
#pragma unroll
    for (int i = 0; i < PIECES; ++i) {
      const int f = feature(i);
      if (!preparing || f >= d) continue;
#pragma unroll
      for (int e = 0; e < E; ++e) zs[row * d + f + e] = z[i][e];
    }
    __syncthreads();
    if (tid < d) {
      float zt = 0.f;
      for (int r = 0; r < S::TOK; ++r) zt += zs[r * d + tid];
      out[d * d + tid] = zt;
      // Values of V below 2^-104 show in S_ij against z_i = sum of phi(k)_i, values of K in z_i against the tokens, and
      // what products of parts lack in sums below 2^-100.
      if (S::REST) {
        const float low = fminf(least[tid], least[128 + tid]);
        if (low < fmaxf(zt * 0x1p-104f, 0x1p-100f) || (zt > 0.f && zt < (float)tiles * (S::TOK * 0x1p-104f))) *odd_flag = 1;
      }
    }
    if (S::REST) {   // (one part each: the products are exact)
      __syncthreads();
      if (*odd_flag) {
        const long long n0 = first * S::TOK, n1 = min(p.N, (first + tiles) * S::TOK);
        state_by_fma<T, ROPE>(k + base, v + base, tab, d, p.sn, n0, n1, zs, out);
      }
    }
  } else if (tid == 0) {
    ctrl->status = LINATTN_ERR_TIMEOUT;
    if (!state) ctrl->gave_up = 1;   // for the sum of partial states
  }
  if (state) {
    cluster_sync();
    // a CTA that gave up has nothing to add: then the state stays as it was
    const bool gave_up = lane < P && lane < 8 && __float_as_int(cluster_load(cluster_address((const void*)abort_flag, lane))) != 0;
    if (!__any_sync(0xffffffffu, gave_up)) {
      const int elems = (int)p.state_elems(), e0 = (int)((long long)c * elems / P), e1 = (int)((long long)(c + 1) * elems / P);
      const long long at = (long long)u * elems;
      uint32_t peer[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) peer[r] = cluster_address(own, r < P ? r : 0);
      for (int e = e0 + tid; e < e1; e += kBlock) {
        float x[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) x[r] = r < P ? cluster_load(peer[r] + 4 * e) : 0.f;
        double total = base_state ? (double)base_state[at + e] : 0.0;
#pragma unroll
        for (int r = 0; r < 8; ++r)
          if (r < P) total += (double)x[r];
        state[at + e] = (float)total;
      }
    }
    cluster_sync();   // nobody leaves while its state is being read
  }
  if (warp == 0) tmem_dealloc(tmem, S::COLS);
}

// ---------------------------------------------------------------- apply
// O^T = S^T phi(Q)^T: the accumulator's lanes are the value features and its columns the tokens of a tile, so that a
// tile of 64 tokens is enough for a whole MMA and three parts of S, two tiles' three parts and the next tile's raw
// pieces fit into shared memory together.
template <typename T, int R, bool ROPE>
struct ApplyShape : Shape<T, R, ROPE> {
  using B = Shape<T, R, ROPE>;
  // One part (bf16): tiles of 128 tokens.  The output is rounded to bf16 there, so one accumulator for the leading products
  // does; three, for short chains, where the output is fp32.
  static constexpr int TOK = B::QK_PARTS == 1 ? 128 : 64;
  static constexpr int LEAD = B::QK_PARTS == 1 ? 1 : 3;
  static constexpr int LANES = kPrepare / TOK;                // threads to a row
  static constexpr int ROUND = B::F32 ? 4 : 2;                // (see flip_of)
  static constexpr int PIECES = ROUND * ((B::DP / B::E + ROUND * LANES - 1) / (ROUND * LANES));   // 16-byte pieces of a row per thread
  static constexpr int FLIP = flip_of(B::E, LANES, PIECES);
  static constexpr int SBOX = B::DP * 128, SPART = B::BOXES * SBOX;   // (lanes from DP on read whatever follows and are ignored)
  static constexpr int S_BYTES = 3 * SPART;
  static constexpr int QBOX = TOK * 128, STAGE = B::QK_PARTS * B::BOXES * QBOX;
  // Three parts of many features: those of a box lie behind one another, so that one MMA takes two of them as 128 columns.  An MMA
  // costs about as much with 64 columns as with 128 (87 to 89 cycles here beside the preparing warps, 65 by itself), and from d = 97 on
  // their number was what the pass waited for (3750 of 4440 cycles a tile to issue 42 of them): four a K step instead of six.
  // 32 760 tokens, apply pass (range of nine runs): 20 heads of 112 187 (186..198) -> 163 us (161..165), 22 of 100 226 -> 208,
  // 18 of 128 176 (175..183) -> 160 (158..165); 4680 tokens 41.6 -> 37.5 and 39.5 -> 37.5.  Smaller heads wait for the draining warps, which
  // read one accumulator more then (80: 212 -> 210, bf16 with rotary factors 405 -> 412, 64: 220 -> 238, 32: 361 -> 402), and keep six.
  static constexpr bool STACK = B::QK_PARTS == 3 && R >= 7;
  static constexpr int QPART = STACK ? QBOX : B::BOXES * QBOX, QBOX_STEP = STACK ? 3 * QBOX : QBOX;
  static constexpr int DEN = (4 * TOK + 128) * 4;
  static constexpr int FIXED = 1024 + S_BYTES + 2 * STAGE + DEN + kBarBytes;
  // a tile's rotations are staged beside its pieces where there is room (not for fp32 at d > 96: loaded where they are used)
  static constexpr bool TAB_STAGED = ROPE && FIXED + PIECES * kPrepare * (16 + (int)sizeof(typename B::Tab)) <= 227 * 1024;
  static constexpr int RAW = PIECES * kPrepare * (16 + (TAB_STAGED ? (int)sizeof(typename B::Tab) : 0));   // one tile as loaded
  static constexpr int FIT = (227 * 1024 - FIXED) / RAW;
  static constexpr int RAW_STAGES = FIT < 1 ? 1 : FIT > 3 ? 3 : FIT;
  static constexpr int OVERRUN = 128 * 128 - SBOX;            // of the last part's last box, when less than that follows
  static constexpr int SMEM = FIXED + (RAW_STAGES * RAW > OVERRUN ? RAW_STAGES * RAW : OVERRUN);
  // TMEM columns: two sets of accumulators.  STACK: two sets of those of the leading products, and one pair for the products of
  // order one (S0 Q1 + S1 Q0) and two (S0 Q2 + S1 Q1 + S2 Q0).
  static constexpr int ACC = TOK, SET = (STACK ? LEAD : LEAD + 1) * ACC, REST = 2 * SET;
  static_assert(2 * SET + (STACK ? 2 * ACC : 0) <= 512, "tensor memory");
  // apply_by_fma's room ends before the barriers and flags, which other threads may still be looking at
  static_assert((B::DP * B::DP + B::DP + 256 * (kBlock + 31) / 32) * 4 <= S_BYTES + 2 * STAGE, "scratch of apply_by_fma");
};

// grid (C, units): tiles [c * tiles / C, (c + 1) * tiles / C) of one unit.
//
// Measured as above: 159 us (163 before early starts), general kernels 866, register-blocked on packed fp32 FMAs 489.  Stamps, cycles of a 64-token tile's
// 3830: the accumulators of order one and two are there once, so a tile's 21 MMAs on them follow the reading of the last tile's:
// read 840, issued 1590, complete 1030 later, 3460 in a chain; beside it the seven leading MMAs (840), the draining warps' stores (2340 of
// their 3180) and the preparing warps (3380).  d = 128: 4520, of which the MMA warp issues for 3240.  bf16, 28 heads of 80:
// 152 us (165 with tiles of 64 tokens and every warp in both roles), general kernels 644.
template <typename T, int R, bool ROPE>
__global__ void __launch_bounds__(kBlock, 1)
split_apply_kernel(const T* __restrict__ q, const float* __restrict__ state, T* __restrict__ o, Problem p, float eps,
                   const __half2* __restrict__ tab, WorkspaceCtrl* ctrl) {
  using A = ApplyShape<T, R, ROPE>;
  using Tab = typename A::Tab;
  constexpr int E = A::E, PIECES = A::PIECES;
  constexpr uint32_t IDESC = make_idesc_bf16(128, A::TOK, false, false);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* s_op = align1024(smem_raw);
  uint8_t* stages = s_op + A::S_BYTES;
  float* den = reinterpret_cast<float*>(stages + 2 * A::STAGE);     // [4][TOK] reciprocals of the denominators
  float* zs = den + 4 * A::TOK;                                     // [128] z
  uint64_t* done = reinterpret_cast<uint64_t*>(zs + 128);           // [2] each, as in the state kernel
  uint64_t* ready = done + 2;
  uint64_t* drained = ready + 2;
  uint64_t* finished = drained + 2;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(finished + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  volatile int* odd_flag = abort_flag + 1;   // the parts are not the values
  uint8_t* raw = reinterpret_cast<uint8_t*>(done) + kBarBytes;
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = p.d, u = blockIdx.y;
  const long long all = (p.N + A::TOK - 1) / A::TOK;
  const long long first = blockIdx.x * all / gridDim.x;
  const int tiles = (int)((blockIdx.x + 1) * all / gridDim.x - first);
  // (Waited for here and not behind the barriers' and tensor memory's set-up: the first pieces were asked for later then, and with more
  // registers spilled in the loops the pass took 168 us and not 159; at the start of the kernel without an early start, 161.)
  wait_for_prior_grids();
  const float* W = behind_wait(state) + (long long)u * p.state_elems();
  const long long base = (long long)(u / p.H) * p.sb + (long long)(u % p.H) * p.sh;
  // preparing: this thread's row of every tile, and its pieces of it
  const int row = (tid % kPrepare) / A::LANES, l = tid % A::LANES;
  auto feature = [&](int i) { return (l + A::LANES * (i ^ (A::FLIP * (row & 1)))) * E; };
  const bool preparing = tid < kPrepare;
  auto raw_q = [&](int st, int i) { return reinterpret_cast<uint4*>(raw + st * A::RAW) + i * kPrepare + tid; };
  auto raw_tab = [&](int st, int i) { return reinterpret_cast<Tab*>(raw + st * A::RAW + PIECES * kPrepare * 16) + i * kPrepare + tid; };
  auto issue = [&](int t) {
    if (t < tiles) {
      const long long n = (first + t) * A::TOK + row;
      const bool live = n < p.N;
      const long long at = live ? n : 0;
      const int st = t % A::RAW_STAGES;
#pragma unroll
      for (int i = 0; i < PIECES; ++i) {
        const int f = feature(i);
        if (f >= d) continue;
        copy_async<16>(raw_q(st, i), q + base + at * p.sn + f, live);
        if (A::TAB_STAGED) copy_async<(int)sizeof(Tab)>(raw_tab(st, i), tab + at * (d / 2) + f / 2, live);
      }
    }
    copy_commit();
  };
  if (preparing) {
#pragma unroll
    for (int t = 0; t < A::RAW_STAGES; ++t) issue(t);
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&done[i], 1); mbar_init(&ready[i], kPrepare); mbar_init(&drained[i], kDrain); }
    mbar_init(finished, 1);
    *abort_flag = *odd_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) { tmem_alloc(tmem_holder, 512); tmem_relinquish(); }
  // padded features of both operands read as zero
  if (d < A::DP)
    for (int i = tid; i < (A::S_BYTES + 2 * A::STAGE) / 16; i += kBlock) reinterpret_cast<uint4*>(s_op)[i] = make_uint4(0, 0, 0, 0);
  if (tid < 128) zs[tid] = tid < d ? W[(long long)d * d + tid] : 0.f;
  __syncthreads();
  uint32_t least = 0xFFFFFFFFu;   // twice the bits of the smallest |S| 2^38, less one (zero is the largest)
  float rest = 0.f;               // NaN if one is not finite
  for (int idx = tid; idx < d * (d / 4); idx += kBlock) {
    const int j = idx / (d / 4), i = (idx - j * (d / 4)) * 4;
    float x[4];
    widen(__ldg(reinterpret_cast<const uint4*>(W + (long long)j * d + i)), x);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float y = x[e] * 0x1p38f;
      least = min(least, 2 * __float_as_uint(y) - 1);
      rest = fmaf(y, 0.f, rest);
    }
    uint32_t unused = 0;
    store_parts<3>(s_op + operand_offset(j, i, A::SBOX), A::SPART, x, unused);
  }
  bool odd = rest != 0.f || least < 2 * __float_as_uint(0x1p-37f) - 1;   // |S| from 2^-75 to 2^90
  fence_proxy_async_smem();   // S and the zeros
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  let_next_grid_start();
  const uint32_t tmem = *tmem_holder;

  if (preparing) {
    // denominators from z_max 2^-50 to z_max 2^35: rows of queries from 2^-57 to 2^35, products with S from 2^-132 to 2^125
    float z_max = 0.f;
    const __half2* const turns = behind_wait(tab);
    for (int i = lane; i < d; i += 32) z_max = fmaxf(z_max, fabsf(zs[i]));
#pragma unroll
    for (int st = 1; st < 32; st *= 2) z_max = fmaxf(z_max, __shfl_xor_sync(0xffffffffu, z_max, st));
    for (int t = 0; t < tiles; ++t) {
      uint8_t* stage = stages + (t & 1) * A::STAGE;
      const int st = t % A::RAW_STAGES;
      uint4 x4[PIECES];   // all reads first, then the tile that takes their place is asked for
      Tab tb[PIECES];
      if (ROPE && !A::TAB_STAGED) {
        const long long n = (first + t) * A::TOK + row;
#pragma unroll
        for (int i = 0; i < PIECES; ++i)
          if (feature(i) < d) tb[i] = __ldg(reinterpret_cast<const Tab*>(turns + (n < p.N ? n : 0) * (d / 2) + feature(i) / 2));
      }
      copy_wait<A::RAW_STAGES - 1>();
#pragma unroll
      for (int i = 0; i < PIECES; ++i) {
        x4[i] = *raw_q(st, i);
        if (A::TAB_STAGED) tb[i] = *raw_tab(st, i);
      }
      issue(t + A::RAW_STAGES);
      // the MMAs that read this stage (the warps below work as a whole, and leave as a whole)
      if (t >= 2 && !__all_sync(0xffffffffu, mbar_wait(&done[t & 1], ((t - 2) >> 1) & 1, abort_flag))) break;
      float dn = 0.f;
#pragma unroll
      for (int i = 0; i < PIECES; ++i) {
        const int f = feature(i);
        if (f >= d) continue;
        float x[E];
        widen(x4[i], x);
#pragma unroll
        for (int e = 0; e < E; e += 4) {
          const float4 z = *reinterpret_cast<const float4*>(zs + f + e);
#pragma unroll
          for (int k = 0; k < 4; ++k) x[e + k] = fmaxf(x[e + k], 0.f);   // phi = ReLU on the queries
          dn = fmaf(x[e], z.x, dn); dn = fmaf(x[e + 1], z.y, dn); dn = fmaf(x[e + 2], z.z, dn); dn = fmaf(x[e + 3], z.w, dn);
        }
        if (ROPE) rotate<E>(x, reinterpret_cast<const __half2*>(&tb[i]));
        uint32_t unused = 0;
        store_parts<A::QK_PARTS>(stage + operand_offset(row, f, A::QBOX_STEP), A::QPART, x, unused);
      }
      __syncwarp();
#pragma unroll
      for (int st2 = 1; st2 < A::LANES; st2 *= 2) dn += __shfl_xor_sync(0xffffffffu, dn, st2);
      odd |= dn != 0.f && !(dn >= z_max * 0x1p-50f && dn <= z_max * 0x1p35f);
      if (l == 0) den[(t & 3) * A::TOK + row] = 1.0f / (dn + eps);   // eps added once, after the dot product
      fence_proxy_async_smem();
      mbar_arrive(&ready[t & 1]);
    }
    copy_wait<0>();
  } else if (warp < kMmaWarp) {
    // accumulator lane = value feature; each of the two warps of a lane quarter takes half of the tokens
    constexpr int HALF = A::TOK / 2;
    const int j = (warp & 3) * 32 + lane, tok0 = ((warp >> 2) & 1) * HALF;
    for (int t = 0; t < tiles; ++t) {
      if (!__all_sync(0xffffffffu, mbar_wait(&done[t & 1], (t >> 1) & 1, abort_flag))) break;   // tcgen05.ld wants whole warps
      tcgen05_fence_after();
      if ((warp & 3) * 32 < d) {
        const uint32_t trow = tmem + (t & 1) * A::SET + ((uint32_t)((warp & 3) * 32) << 16) + tok0;
        const uint32_t rrow = tmem + A::REST + ((uint32_t)((warp & 3) * 32) << 16) + tok0;
        const float* rden = den + (t & 3) * A::TOK + tok0;
        const long long n0 = (first + t) * A::TOK + tok0;
        const int live = j < d ? (int)min((long long)HALF, p.N - n0) : 0;
        T* out = o + base + n0 * p.sn + j;
        constexpr int LEADS = R < A::LEAD ? R : A::LEAD;
        auto read = [&](int g, float (&num)[8]) {   // numerators of tokens 8 g .. 8 g + 7
          uint32_t a[A::LEAD + 2][8];
#pragma unroll
          for (int s = 0; s < LEADS; ++s) tmem_ld_x8(trow + s * A::ACC + 8 * g, a[s]);
          if (A::STACK) {
            tmem_ld_x8(rrow + 8 * g, a[A::LEAD]);
            tmem_ld_x8(rrow + A::ACC + 8 * g, a[A::LEAD + 1]);
          } else {
            tmem_ld_x8(trow + A::LEAD * A::ACC + 8 * g, a[A::LEAD]);
          }
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            num[x] = __uint_as_float(a[0][x]);
#pragma unroll
            for (int s = 1; s < LEADS; ++s) num[x] += __uint_as_float(a[s][x]);
            num[x] += A::STACK ? __uint_as_float(a[A::LEAD + 1][x]) + __uint_as_float(a[A::LEAD][x]) : __uint_as_float(a[A::LEAD][x]);
          }
        };
        auto write = [&](int g, const float (&num)[8]) {
          float wild = 0.f;   // NaN if a numerator is not finite: queries where z is zero, which no denominator sees, have no bounds
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            if (8 * g + x < live) {
              store_value(out, num[x] * rden[8 * g + x]);
              wild = fmaf(num[x], 0.f, wild);
            }
            out += p.sn;
          }
          if (wild != 0.f) *odd_flag = 1;
        };
        if constexpr (A::STACK) {   // the next tile's MMAs wait for the accumulators: all read, and handed back, before the first is stored
          float num[HALF / 8][8];
#pragma unroll
          for (int g = 0; g < HALF / 8; ++g) read(g, num[g]);
          tcgen05_fence_before();
          mbar_arrive(&drained[t & 1]);
#pragma unroll
          for (int g = 0; g < HALF / 8; ++g) write(g, num[g]);
          continue;
        } else {
#pragma unroll
          for (int g = 0; g < HALF / 8; ++g) {
            float num[8];
            read(g, num);
            write(g, num);
          }
        }
      }
      tcgen05_fence_before();
      mbar_arrive(&drained[t & 1]);
    }
  } else if (lane == 0) {
    int t = 0;
    bool issued = false;   // MMAs of a tile that was not completed
    for (; t < tiles; ++t) {
      if (t >= 2 && !mbar_wait(&drained[t & 1], ((t - 2) >> 1) & 1, abort_flag)) break;
      if (!mbar_wait(&ready[t & 1], (t >> 1) & 1, abort_flag)) break;
      tcgen05_fence_after();
      const uint64_t a0 = make_smem_desc_sw128(smem_u32(s_op), 16, 1024);   // offsets are added as in the state kernel
      const uint64_t b0 = make_smem_desc_sw128(smem_u32(stages + (t & 1) * A::STAGE), 16, 1024);
      const uint32_t set = tmem + (t & 1) * A::SET;
      auto mma = [&](int kk, int ps, int pq, uint32_t acc, uint32_t idesc, bool add) {
        umma_bf16(acc, a0 + (ps * A::SPART + (kk >> 2) * A::SBOX + (kk & 3) * 32) / 16,
                  b0 + (pq * A::QPART + (kk >> 2) * A::QBOX_STEP + (kk & 3) * 32) / 16, idesc, add ? 1u : 0u);
      };
      if constexpr (A::STACK) {
        constexpr uint32_t WIDE = make_idesc_bf16(128, 2 * A::TOK, false, false);
#pragma unroll
        for (int kk = 0; kk < R; ++kk) mma(kk, 0, 0, set + (kk % A::LEAD) * A::ACC, IDESC, kk >= A::LEAD);
        issued = true;
        if (t > 0 && !mbar_wait(&drained[(t - 1) & 1], ((t - 1) >> 1) & 1, abort_flag)) break;   // the pair
        tcgen05_fence_after();
        const uint32_t rest = tmem + A::REST;
#pragma unroll
        for (int kk = 0; kk < R; ++kk) {
          mma(kk, 0, 1, rest, WIDE, kk > 0);                 // S0 [Q1 | Q2]
          mma(kk, 1, 0, rest, WIDE, true);                   // S1 [Q0 | Q1]
          mma(kk, 2, 0, rest + A::ACC, IDESC, true);         // S2 Q0
        }
      } else {
        bool add = false;
#pragma unroll
        for (int order = 2; order >= 1; --order)   // smallest first
#pragma unroll
          for (int pq = order; pq >= 0; --pq) {
            if (pq >= A::QK_PARTS) continue;
#pragma unroll
            for (int kk = 0; kk < R; ++kk) { mma(kk, order - pq, pq, set + A::LEAD * A::ACC, IDESC, add); add = true; }
          }
#pragma unroll
        for (int kk = 0; kk < R; ++kk) mma(kk, 0, 0, set + (kk % A::LEAD) * A::ACC, IDESC, kk >= A::LEAD);
      }
      umma_commit(&done[t & 1]);
    }
    if (t > 0 || issued) umma_commit(finished); else mbar_arrive(finished);
  }
  if (odd) *odd_flag = 1;
  __syncthreads();
  const bool aborted = *abort_flag != 0;
  if (aborted) let_finish(finished);
  if (!aborted && *odd_flag) {
    const long long n0 = first * A::TOK, n1 = min(p.N, (first + tiles) * A::TOK);
    apply_by_fma<T, ROPE>(q + base, W, o + base, tab, d, p.sn, n0, n1, eps, reinterpret_cast<float*>(s_op));
  }
  if (aborted && tid == 0) ctrl->status = LINATTN_ERR_TIMEOUT;
  if (warp == 0) { tcgen05_fence_after(); tmem_dealloc(tmem, 512); }
}

// ---------------------------------------------------------------- host side
int sms() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!cached[dev]) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    cached[dev] = n;
  }
  return cached[dev];
}

template <typename K>
cudaError_t allow_smem(K kernel, int bytes, bool (&done)[64]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (done[dev]) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

// How many pieces a unit's tiles are cut into, up to `most`: the fewest waves of CTAs times what a CTA takes, `fixed`
// tiles of which it takes whatever its share.
int pieces(long long tiles, int units, int slots, long long most, double fixed) {
  const long long few = (4ll * slots + units - 1) / units;   // four waves: beyond that the last one is small anyway
  if (most > few) most = few;
  if (most > tiles) most = tiles;
  long long best = 1;
  double cost = 0;
  for (long long c = 1; c <= most; ++c) {
    const double now = (double)((c * units + slots - 1) / slots) * ((double)((tiles + c - 1) / c) + fixed);
    if (c == 1 || now < cost) { best = c; cost = now; }
  }
  return (int)best;
}

// Clusters of c CTAs of `kernel` that fit on the device together (0: none), c = 1..8.
template <typename K>
int clusters_at_once(K kernel, int smem, int c, int (&cached)[64][9]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!cached[dev][c]) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)c, 1, 1};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(c); cfg.blockDim = dim3(kBlock); cfg.dynamicSmemBytes = smem;
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }   // (asked again next time)
    cached[dev][c] = n > 0 ? n : -1;
  }
  return cached[dev][c] > 0 ? cached[dev][c] : 0;
}

// *P = 0: the state is complete; otherwise *P partial states per unit are to be summed.
template <typename T, int R, bool ROPE>
cudaError_t launch_state(const Problem& p, const void* k, const void* v, const float* base, float* state, float* partials,
                         const __half2* tab, int* P, WorkspaceCtrl* ctrl, cudaStream_t stream) {
  using S = StateShape<T, R, ROPE>;
  static_assert(S::SMEM <= 227 * 1024, "shared memory of the state kernel");
  static bool done[64] = {false};
  static int fits[64][9] = {{0}};
  auto kernel = split_state_kernel<T, R, ROPE>;
  const cudaError_t e = allow_smem(kernel, S::SMEM, done);
  if (e != cudaSuccess) return e;
  const long long tiles = (p.N + S::TOK - 1) / S::TOK;
  // In tiles: a CTA costs six whatever its share, the sum of partial states (a kernel of its own) one more than a cluster's.
  // Measured, cached step, fp32, 20 heads of 112, cluster against partial states: 300 tokens 24.9 against 33.3 us, 512 29.9
  // against 43.8, 1200 37.6 against 43.7, 4680 75.9 against 73.9; forward of 3000 tokens, 35 heads of 64: 62.5 against 57.8.
  // (Without early starts, which take 2 us off a call of either.)
  *P = pieces(tiles, p.units(), sms(), fma_chunks(p.N), 6.0);
  const double apart = (double)(((long long)*P * p.units() + sms() - 1) / sms()) * ((double)((tiles + *P - 1) / *P) + 6.0) + 1.0;
  int together = 0;
  double cost = apart;
  for (int c = 1; c <= 8 && c <= tiles; ++c) {
    const int at_once = clusters_at_once(kernel, S::SMEM, c, fits);
    if (!at_once) continue;
    const double now = (double)((p.units() + at_once - 1) / at_once) * ((double)((tiles + c - 1) / c) + 6.0);
    if (now < cost) { together = c; cost = now; }
  }
  bool early = true;
  if (together > 2 && together % 2)
    early = clusters_start_early(together, p.units(), clusters_at_once(kernel, S::SMEM, together, fits), clusters_at_once(kernel, S::SMEM, together + 1, fits),
                                 (p.N + 32ll * together - 1) / (32ll * together));
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)(together ? together : 1), 1, 1};
  at[1] = early_start();
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(together ? together : *P, p.units());
  cfg.blockDim = dim3(kBlock); cfg.dynamicSmemBytes = S::SMEM; cfg.stream = stream;
  cfg.attrs = at; cfg.numAttrs = early ? 2 : 1;
  const cudaError_t st = cudaLaunchKernelEx(&cfg, kernel, (const T*)k, (const T*)v, p, together ? together : *P, partials, base,
                                            together ? state : (float*)nullptr, tab, ctrl);
  if (st != cudaSuccess) { cudaGetLastError(); return st; }
  if (together) *P = 0;
  count_launches(1);
  return cudaSuccess;
}

template <typename T, int R, bool ROPE>
cudaError_t launch_apply(const Problem& p, const void* q, const float* state, void* o, float eps, const __half2* tab,
                         WorkspaceCtrl* ctrl, cudaStream_t stream) {
  using A = ApplyShape<T, R, ROPE>;
  static_assert(A::SMEM <= 227 * 1024, "shared memory of the apply kernel");
  static bool done[64] = {false};
  const cudaError_t e = allow_smem(split_apply_kernel<T, R, ROPE>, A::SMEM, done);
  if (e != cudaSuccess) return e;
  const int C = pieces((p.N + A::TOK - 1) / A::TOK, p.units(), sms(), 1ll << 30, 4.0);
  const cudaError_t st = launch_early(split_apply_kernel<T, R, ROPE>, dim3(C, p.units()), dim3(kBlock), A::SMEM, stream, (const T*)q, state, (T*)o, p,
                                      eps, tab, ctrl);
  if (st != cudaSuccess) { cudaGetLastError(); return st; }
  count_launches(1);
  return cudaSuccess;
}

#define LINATTN_SPLIT(FN, T, ROPE, ...)              \
  switch ((p.d + 15) / 16) {                         \
    case 2: return FN<T, 2, ROPE>(__VA_ARGS__);      \
    case 3: return FN<T, 3, ROPE>(__VA_ARGS__);      \
    case 4: return FN<T, 4, ROPE>(__VA_ARGS__);      \
    case 5: return FN<T, 5, ROPE>(__VA_ARGS__);      \
    case 6: return FN<T, 6, ROPE>(__VA_ARGS__);      \
    case 7: return FN<T, 7, ROPE>(__VA_ARGS__);      \
    default: return FN<T, 8, ROPE>(__VA_ARGS__);     \
  }

}  // namespace

// These kernels read rows in 16-byte pieces and the rotations of a piece in one load; everything else (odd head dims,
// unaligned views) takes the general kernels, and so do head dims up to 16, whose tiles are too small for what a tile
// costs here (2000 tokens: 100 heads of 8 in bf16 71 against 47 us, 140 heads of 16 in fp32 95 against 69 us; from
// d = 24 on these kernels win at every size measured, 4000 tokens, 70 heads of 32 in fp32: 103 against 135 us).
bool split_ok(const Problem& p, const void* a, const void* b, const __half2* rope) {
  const int per = p.dtype == LINATTN_F32 ? 4 : 8;
  const uintptr_t tab_align = p.dtype == LINATTN_F32 ? 7 : 15;
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0 && p.d > 16 && p.d % per == 0 && p.sb % per == 0 &&
         p.sn % per == 0 && p.sh % per == 0 && (reinterpret_cast<uintptr_t>(rope) & tab_align) == 0;
}

cudaError_t split_state(const Problem& p, const void* k, const void* v, const float* base, float* state, float* partials,
                        const __half2* rope, int* P, WorkspaceCtrl* ctrl, cudaStream_t stream) {
  if (p.dtype == LINATTN_F32) {
    if (rope) { LINATTN_SPLIT(launch_state, float, true, p, k, v, base, state, partials, rope, P, ctrl, stream) }
    LINATTN_SPLIT(launch_state, float, false, p, k, v, base, state, partials, rope, P, ctrl, stream)
  }
  if (rope) { LINATTN_SPLIT(launch_state, __nv_bfloat16, true, p, k, v, base, state, partials, rope, P, ctrl, stream) }
  LINATTN_SPLIT(launch_state, __nv_bfloat16, false, p, k, v, base, state, partials, rope, P, ctrl, stream)
}

cudaError_t split_apply(const Problem& p, const void* q, const float* state, void* o, float eps, const __half2* rope,
                        WorkspaceCtrl* ctrl, cudaStream_t stream) {
  if (p.dtype == LINATTN_F32) {
    if (rope) { LINATTN_SPLIT(launch_apply, float, true, p, q, state, o, eps, rope, ctrl, stream) }
    LINATTN_SPLIT(launch_apply, float, false, p, q, state, o, eps, rope, ctrl, stream)
  }
  if (rope) { LINATTN_SPLIT(launch_apply, __nv_bfloat16, true, p, q, state, o, eps, rope, ctrl, stream) }
  LINATTN_SPLIT(launch_apply, __nv_bfloat16, false, p, q, state, o, eps, rope, ctrl, stream)
}

}  // namespace linattn
