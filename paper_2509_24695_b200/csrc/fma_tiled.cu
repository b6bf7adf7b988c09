// Register-blocked fp32 kernels of the FMA path: fp32 tensors, and the bf16 head dims the tensor-core kernel does not
// take, wherever rows can be read in 16-byte pieces (fma_tiled_ok).  fp32 arithmetic throughout, as in fma_kernels.cu,
// which keeps every other shape.
//
// Both contractions are bound by the fp32 pipe here (d/2 multiply-adds per byte of fp32 input: a fifth of the HBM rate
// at its peak), so what counts is how few other instructions and shared-memory reads go with a multiply-add: every
// thread owns a large register tile of the result, fp32 FMAs are issued in pairs (fma.rn.f32x2: the same rate as the
// scalar form on this part, with half the issue slots), and operands come from shared memory already widened, rectified,
// rotated and, where both halves of a pair need the same value, doubled.
//
// Measured times are with the kernels below; the fp32 pipe gives 63 (packed) to 72 TFLOP/s on this part.
#include "common.cuh"

namespace linattn {
namespace {

typedef unsigned long long u64;

__device__ __forceinline__ void fma2_acc(u64& acc, u64 a, u64 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ u64 twice(float x) {
  u64 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 halves(u64 r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}

// 16 bytes of a row as floats
template <typename T>
struct Chunk;
template <>
struct Chunk<float> {
  static constexpr int E = 4;
  using Tab = uint2;   // the (cos, sin) fp16 pairs of its feature pairs
  static __device__ __forceinline__ void widen(const uint4& r, float (&x)[4]) {
    x[0] = __uint_as_float(r.x); x[1] = __uint_as_float(r.y); x[2] = __uint_as_float(r.z); x[3] = __uint_as_float(r.w);
  }
};
template <>
struct Chunk<__nv_bfloat16> {
  static constexpr int E = 8;
  using Tab = uint4;
  static __device__ __forceinline__ void widen(const uint4& r, float (&x)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { x[2 * i] = __uint_as_float(w[i] << 16); x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
  }
};

// (a, b) -> (a c - b s, b c + a s) for every feature pair of the chunk; `tab` holds the (cos, sin) fp16 pairs
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

// Private copies into shared memory: the thread that issued them is the only one to read them.
template <int BYTES>
__device__ __forceinline__ void copy_async(void* smem_dst, const void* src, bool live) {   // not live: zeros
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(live ? 8 : 0) : "memory");
}

// ---------------------------------------------------------------- state
constexpr int kTokens = 32;   // tokens staged per iteration

// R = ceil(d / 16).  A group of threads owns one whole state, TI x TJ of it per thread; the groups of a CTA take
// different tokens of every staged tile and are added up at the end.  The larger the register tile, the fewer
// shared-memory reads per FMA, until it no longer fits: 2R x 2R with 64 threads to a state (256 threads a CTA), except
// 7 x 14 with 128 threads to a state and 512 a CTA for d in 97..112 (14 x 14 spills: 615 against 492 us for the state
// of 32 760 tokens, 20 heads of 112; the same smaller tile is 7 to 21 % slower at the smaller head dims) and 8 x 16 for
// d > 112.  Before (fma_kernels.cu, 7 x 7 per thread, scalar loads): 1051 us.
template <typename T, int R, bool ROPE>
struct StateShape {
  static constexpr bool PAIRS = R != 7;   // a thread's key features come in pairs: one 16-byte load for two doubled values
  static constexpr int THREADS = R == 7 ? 512 : 256;
  static constexpr int TI = R < 7 ? 2 * R : R, TJ = 2 * R;
  static constexpr int GX = R < 7 ? 8 : 16, GY = 8;
  static constexpr int GROUP = GX * GY, GROUPS = THREADS / GROUP;
  static constexpr int DP = 16 * R;                              // features with padding
  static constexpr int E = Chunk<T>::E;
  static constexpr int ROWS = THREADS / (DP / E);          // rows one pass of the CTA stages (at least)
  static constexpr int PASSES = (kTokens + ROWS - 1) / ROWS;
  static constexpr int TAB = ROPE ? (int)sizeof(typename Chunk<T>::Tab) : 0;
  static constexpr int RAW = PASSES * THREADS * (32 + TAB);      // one stage: K, V and table pieces as loaded
  static constexpr int TILE = kTokens * DP * (8 + 4);                  // one tile: K doubled, V
  static constexpr int PITCH = DP + 4;                                 // rows of the state while the groups are added up
  static constexpr int Z_FLOATS = THREADS * E;
  static constexpr int LOOP = 2 * RAW + 2 * TILE, SUM = (DP * PITCH + Z_FLOATS) * 4;
  static constexpr int SMEM = LOOP > SUM ? LOOP : SUM;
  static constexpr int CTAS = R >= 5 || SMEM > 113 * 1024 ? 1 : 2;   // per SM
  static __device__ __forceinline__ int key(int ti, int r) { return PAIRS ? 2 * ti + 2 * GX * (r / 2) + r % 2 : ti + GX * r; }
};

// grid (P, units): partial state of one token range of one unit, in the library's layout.
template <typename T, int R, bool ROPE>
__global__ void __launch_bounds__(StateShape<T, R, ROPE>::THREADS, StateShape<T, R, ROPE>::CTAS)
fma_tiled_state(const T* __restrict__ k, const T* __restrict__ v, Problem p, int P, float* __restrict__ partials,
                const __half2* __restrict__ tab) {
  using S = StateShape<T, R, ROPE>;
  using Tab = typename Chunk<T>::Tab;
  constexpr int E = S::E, DP = S::DP, TI = S::TI, TJ = S::TJ, THREADS = S::THREADS;
  extern __shared__ __align__(16) uint8_t smem[];
  const int d = p.d, tid = (int)threadIdx.x;
  const int u = blockIdx.y, c = blockIdx.x;
  const long long chunk = (p.N + P - 1) / P;
  const long long n_begin = min(p.N, c * chunk), n_end = min(p.N, n_begin + chunk);
  const int tiles = (int)((n_end - n_begin + kTokens - 1) / kTokens);

  // staging: this thread always has the same 16-byte column, so that its plain phi(k) add up to a share of z
  const int cpr = d / E, rows = THREADS / cpr;
  const int col = tid % cpr, row0 = tid / cpr;
  const bool staging = row0 < rows;
  const long long base = (long long)(u / p.H) * p.sb + (long long)(u % p.H) * p.sh + (long long)col * E;
  auto raw_k = [&](int st, int ps) { return reinterpret_cast<uint4*>(smem + st * S::RAW) + (2 * ps) * THREADS + tid; };
  auto raw_tab = [&](int st, int ps) {
    return reinterpret_cast<Tab*>(smem + st * S::RAW + S::PASSES * THREADS * 32) + ps * THREADS + tid;
  };
  auto k_of = [&](int buf) { return reinterpret_cast<float*>(smem + 2 * S::RAW + buf * S::TILE); };   // [token][DP] pairs
  auto v_of = [&](int buf) { return k_of(buf) + kTokens * DP * 2; };                                  // [token][DP]

  auto issue = [&](int t, int st) {
    if (staging) {
#pragma unroll
      for (int ps = 0; ps < S::PASSES; ++ps) {
        const int row = row0 + ps * rows;
        if (row >= kTokens) break;
        const long long n = n_begin + (long long)t * kTokens + row;
        const bool live = n < n_end;
        const long long off = live ? base + n * p.sn : base;
        copy_async<16>(raw_k(st, ps), k + off, live);
        copy_async<16>(raw_k(st, ps) + THREADS, v + off, live);
        if (ROPE) copy_async<(int)sizeof(Tab)>(raw_tab(st, ps), tab + ((live ? n : 0) * (d / 2) + col * (E / 2)), live);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float z[E];
#pragma unroll
  for (int e = 0; e < E; ++e) z[e] = 0.f;
  auto convert = [&](int st, int buf) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (!staging) return;
#pragma unroll
    for (int ps = 0; ps < S::PASSES; ++ps) {
      const int row = row0 + ps * rows;
      if (row >= kTokens) break;
      float x[E];
      Chunk<T>::widen(*raw_k(st, ps), x);
#pragma unroll
      for (int e = 0; e < E; ++e) { x[e] = fmaxf(x[e], 0.f); z[e] += x[e]; }   // phi = ReLU on the keys; z from the plain ones
      if (ROPE) {
        const Tab t4 = *raw_tab(st, ps);
        rotate<E>(x, reinterpret_cast<const __half2*>(&t4));
      }
      float4* kd = reinterpret_cast<float4*>(k_of(buf) + (row * DP + col * E) * 2);
#pragma unroll
      for (int e = 0; e < E; e += 2) kd[e / 2] = make_float4(x[e], x[e], x[e + 1], x[e + 1]);
      Chunk<T>::widen(*(raw_k(st, ps) + THREADS), x);
      float4* vd = reinterpret_cast<float4*>(v_of(buf) + row * DP + col * E);
#pragma unroll
      for (int e = 0; e < E; e += 4) vd[e / 4] = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
    }
  };

  if (d < DP) {   // padded features stay zero: the staging never writes them
    for (int i = tid; i < 2 * S::TILE / 16; i += THREADS) reinterpret_cast<uint4*>(smem + 2 * S::RAW)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
  }
  const int g = tid / S::GROUP, tg = tid % S::GROUP, ti = tg / S::GY, tj = tg % S::GY;
  u64 acc[TI][TJ / 2];   // (i; j, j + 1) with i = S::key(ti, r), j = 2 tj + 16 s
#pragma unroll
  for (int r = 0; r < TI; ++r)
#pragma unroll
    for (int s = 0; s < TJ / 2; ++s) acc[r][s] = 0;

  issue(0, 0);
  convert(0, 0);
  if (tiles > 1) issue(1, 1);
  __syncthreads();
  for (int t = 0; t < tiles; ++t) {
    // tile t + 1 has had the whole of tile t - 1's arithmetic to arrive; tile t + 2 gets tile t's
    if (t + 1 < tiles) convert((t + 1) & 1, (t + 1) & 1);
    if (t + 2 < tiles) issue(t + 2, t & 1);
    const float* kt = k_of(t & 1) + (size_t)(g * (kTokens / S::GROUPS)) * DP * 2 + 2 * S::key(ti, 0);
    const float* vt = v_of(t & 1) + (size_t)(g * (kTokens / S::GROUPS)) * DP + 2 * tj;
#pragma unroll 2
    for (int n = 0; n < kTokens / S::GROUPS; ++n, kt += 2 * DP, vt += DP) {
      u64 b[TJ / 2];
#pragma unroll
      for (int s = 0; s < TJ / 2; ++s) b[s] = *reinterpret_cast<const u64*>(vt + 16 * s);
#pragma unroll
      for (int r = 0; r < TI; r += S::PAIRS ? 2 : 1) {
        const float* at = kt + 2 * S::GX * r;
        ulonglong2 a;
        if (S::PAIRS) a = *reinterpret_cast<const ulonglong2*>(at);
        else a.x = *reinterpret_cast<const u64*>(at);
#pragma unroll
        for (int s = 0; s < TJ / 2; ++s) {
          fma2_acc(acc[r][s], a.x, b[s]);
          if (S::PAIRS) fma2_acc(acc[r + (S::PAIRS ? 1 : 0)][s], a.y, b[s]);
        }
      }
    }
    __syncthreads();
  }

  // add the groups up in their order, then store W[j][i] = S[i][j] and W[d][i] = z[i]
  float* sum = reinterpret_cast<float*>(smem);
  float* zs = sum + DP * S::PITCH;
#pragma unroll 1
  for (int gg = 0; gg < S::GROUPS; ++gg) {
    if (g == gg) {
#pragma unroll
      for (int s = 0; s < TJ / 2; ++s)
#pragma unroll
        for (int r = 0; r < TI; ++r) {
          const float2 x = halves(acc[r][s]);
          float* at = sum + (2 * tj + 16 * s) * S::PITCH + S::key(ti, r);
          at[0] = gg == 0 ? x.x : at[0] + x.x;
          at[S::PITCH] = gg == 0 ? x.y : at[S::PITCH] + x.y;
        }
    }
    if (gg == 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) zs[tid * E + e] = z[e];   // thread (row0, col): floats row0 * d + col * E ..
    }
    __syncthreads();
  }
  float* out = partials + ((long long)u * P + c) * p.state_elems();
  for (int idx = tid; idx < d * d; idx += THREADS) out[idx] = sum[(idx / d) * S::PITCH + idx % d];
  if (tid < d) {
    float zt = 0.f;
    for (int r = 0; r < rows; ++r) zt += zs[r * d + tid];
    out[(long long)d * d + tid] = zt;
  }
}

// ---------------------------------------------------------------- apply
// A CTA keeps S of its unit in shared memory and walks tiles of NT tokens; a thread owns TN tokens x TJ value features.
// Two CTAs per SM (one at d > 112): one loads and rectifies its tile while the other computes.  32 760 tokens, 20 heads
// of 112, fp32: 489 us (34 TFLOP/s; an instruction per warp every 4.4 cycles with two warps to a scheduler), before
// (fma_kernels.cu, 4 x 7 per thread, S read again for every 64 tokens) 866 us.
template <int R>
struct ApplyShape {
  static constexpr int TN = 8, TJ = 2 * R;
  static constexpr int GN = R < 8 ? 16 : 32, GJ = 8;
  static constexpr int THREADS = GN * GJ, NT = TN * GN;
  static constexpr int DP = 16 * R;
  static constexpr int SP = DP + 2;   // pitch of S: transposing it in conflicts two ways at most
  static constexpr int QP = DP + 4;   // pitch of the tile: rows of one warp's reads and of the row-wise pass miss one another
  static constexpr int SMEM = (DP * SP + 128 + NT * QP + NT) * 4;
  static constexpr int CTAS = R < 8 ? 2 : 1;
};

__device__ __forceinline__ void store_pair(float* o, float a, float b) { *reinterpret_cast<float2*>(o) = make_float2(a, b); }
__device__ __forceinline__ void store_pair(__nv_bfloat16* o, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(o) = __floats2bfloat162_rn(a, b);
}

// grid (C, units): CTA c takes tiles [c * tiles / C, (c + 1) * tiles / C) of its unit.
template <typename T, int R, bool ROPE>
__global__ void __launch_bounds__(ApplyShape<R>::THREADS, ApplyShape<R>::CTAS)
fma_tiled_apply(const T* __restrict__ q, const float* __restrict__ state, T* __restrict__ o, Problem p, float eps,
                const __half2* __restrict__ tab) {
  using A = ApplyShape<R>;
  using Tab = typename Chunk<T>::Tab;
  constexpr int E = Chunk<T>::E, TN = A::TN, TJ = A::TJ, NT = A::NT, THREADS = A::THREADS;
  constexpr int LOADS = 14;   // 16-byte loads a thread has in flight
  extern __shared__ __align__(16) uint8_t smem[];
  float* Ss = reinterpret_cast<float*>(smem);   // [d][SP]: Ss[i][j] = S[i][j], padded columns zero
  float* Qs = Ss + A::DP * A::SP + 128;         // [NT][QP]: phi(q) of the tile (rotated with ROPE)
  float* zs = Ss + A::DP * A::SP;               // [d]
  float* den = Qs + NT * A::QP;                 // [NT]
  const int d = p.d, tid = (int)threadIdx.x, u = blockIdx.y;
  const float* W = state + (long long)u * p.state_elems();
  for (int idx = tid; idx < d * d; idx += THREADS) Ss[(idx % d) * A::SP + idx / d] = W[idx];
  for (int idx = tid; idx < d * (A::DP - d); idx += THREADS) Ss[(idx % d) * A::SP + d + idx / d] = 0.f;
  if (tid < d) zs[tid] = W[(long long)d * d + tid];

  const long long ubase = (long long)(u / p.H) * p.sb + (long long)(u % p.H) * p.sh;
  const long long tiles = (p.N + NT - 1) / NT;
  const long long t0 = blockIdx.x * tiles / gridDim.x, t1 = (blockIdx.x + 1) * tiles / gridDim.x;
  const int cpr = d / E, total = NT * cpr;
  const int tn = tid / A::GJ, tj = tid % A::GJ;
  for (long long t = t0; t < t1; ++t) {
    const long long n0 = t * NT;
    // rows in, rectified, consecutive threads on consecutive pieces
    for (int first = tid; first < total; first += LOADS * THREADS) {
      uint4 x[LOADS];
#pragma unroll
      for (int l = 0; l < LOADS; ++l) {
        const int idx = first + l * THREADS, n = idx / cpr, cc = idx - n * cpr;
        x[l] = make_uint4(0, 0, 0, 0);
        if (idx < total && n0 + n < p.N) x[l] = __ldcs(reinterpret_cast<const uint4*>(q + ubase + (n0 + n) * p.sn + cc * E));
      }
#pragma unroll
      for (int l = 0; l < LOADS; ++l) {
        const int idx = first + l * THREADS, n = idx / cpr, cc = idx - n * cpr;
        if (idx >= total) break;
        float f[E];
        Chunk<T>::widen(x[l], f);
#pragma unroll
        for (int e = 0; e < E; e += 4)
          *reinterpret_cast<float4*>(Qs + n * A::QP + cc * E + e) =
              make_float4(fmaxf(f[e], 0.f), fmaxf(f[e + 1], 0.f), fmaxf(f[e + 2], 0.f), fmaxf(f[e + 3], 0.f));
      }
    }
    __syncthreads();
    // one thread per row: the denominator from the plain phi(q), then (ROPE) the rotation in place
    if (tid < NT) {
      float* row = Qs + tid * A::QP;
      float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
      const long long n = n0 + tid < p.N ? n0 + tid : p.N - 1;
#pragma unroll 4
      for (int cc = 0; cc < cpr; ++cc) {
        float f[E];
#pragma unroll
        for (int e = 0; e < E; e += 4) {
          const float4 a = *reinterpret_cast<const float4*>(row + cc * E + e);
          const float4 b = *reinterpret_cast<const float4*>(zs + cc * E + e);
          s4.x = fmaf(a.x, b.x, s4.x); s4.y = fmaf(a.y, b.y, s4.y); s4.z = fmaf(a.z, b.z, s4.z); s4.w = fmaf(a.w, b.w, s4.w);
          f[e] = a.x; f[e + 1] = a.y; f[e + 2] = a.z; f[e + 3] = a.w;
        }
        if (ROPE) {
          const Tab t4 = __ldg(reinterpret_cast<const Tab*>(tab + n * (d / 2) + cc * (E / 2)));
          rotate<E>(f, reinterpret_cast<const __half2*>(&t4));
#pragma unroll
          for (int e = 0; e < E; e += 4)
            *reinterpret_cast<float4*>(row + cc * E + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
        }
      }
      den[tid] = ((s4.x + s4.y) + (s4.z + s4.w)) + eps;   // eps added once, after the dot product
    }
    __syncthreads();
    u64 acc[TN][TJ / 2];   // tokens tn + GN r; value features 2 tj + 16 s, + 1
#pragma unroll
    for (int r = 0; r < TN; ++r)
#pragma unroll
      for (int s = 0; s < TJ / 2; ++s) acc[r][s] = 0;
    const float* qrow = Qs + tn * A::QP;
    const float* srow = Ss + 2 * tj;
#pragma unroll 1
    for (int i = 0; i < d; i += 4, qrow += 4, srow += 4 * A::SP) {
      float4 a[TN];
#pragma unroll
      for (int r = 0; r < TN; ++r) a[r] = *reinterpret_cast<const float4*>(qrow + r * A::GN * A::QP);
#pragma unroll
      for (int ii = 0; ii < 4; ++ii) {
        u64 b[TJ / 2];
#pragma unroll
        for (int s = 0; s < TJ / 2; ++s) b[s] = *reinterpret_cast<const u64*>(srow + ii * A::SP + 16 * s);
#pragma unroll
        for (int r = 0; r < TN; ++r) {
          const u64 aa = twice(ii == 0 ? a[r].x : ii == 1 ? a[r].y : ii == 2 ? a[r].z : a[r].w);
#pragma unroll
          for (int s = 0; s < TJ / 2; ++s) fma2_acc(acc[r][s], aa, b[s]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < TN; ++r) {
      const int row = tn + A::GN * r;
      if (n0 + row >= p.N) break;
      const float dn = den[row];
      T* out = o + ubase + (n0 + row) * p.sn + 2 * tj;
#pragma unroll
      for (int s = 0; s < TJ / 2; ++s) {
        const float2 x = halves(acc[r][s]);
        if (2 * tj + 16 * s < d) store_pair(out + 16 * s, x.x / dn, x.y / dn);
      }
    }
    __syncthreads();   // the next tile overwrites Qs and den
  }
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

// How many pieces a unit's `work` is cut into, from `least` to `most`: the fewest waves of CTAs times what a CTA takes,
// `fixed` (in units of work) of which it takes whatever its share.
int pieces(long long work, int units, int slots, long long least, long long most, double fixed) {
  long long best = least;
  double cost = 0;
  for (long long c = least; c <= most; ++c) {
    const double waves = (double)((c * units + slots - 1) / slots);
    const double now = waves * ((double)((work + c - 1) / c) + fixed);
    if (c == least || now < cost) { best = c; cost = now; }
  }
  return (int)best;
}

template <typename T, int R, bool ROPE>
cudaError_t launch_state(const Problem& p, const void* k, const void* v, float* partials, const __half2* tab, int* P,
                         cudaStream_t stream) {
  using S = StateShape<T, R, ROPE>;
  static bool done[64] = {false};
  const cudaError_t e = allow_smem(fma_tiled_state<T, R, ROPE>, S::SMEM, done);
  if (e != cudaSuccess) return e;
  // one accumulator adds up at most 512 tokens (a CTA's groups share its tokens) where the workspace has room for that
  // many partial states: no longer chains of fp32 additions than fma_kernels.cu has
  const long long most = fma_chunks(p.N), per = 512ll * S::GROUPS;
  const long long least = (p.N + per - 1) / per;
  *P = pieces(p.N, p.units(), sms() * S::CTAS, least < most ? least : most, most, 100.0);
  fma_tiled_state<T, R, ROPE><<<dim3(*P, p.units()), S::THREADS, S::SMEM, stream>>>((const T*)k, (const T*)v, p, *P, partials, tab);
  count_launches(1);
  return cudaGetLastError();
}

template <typename T, int R, bool ROPE>
cudaError_t launch_apply(const Problem& p, const void* q, const float* state, void* o, float eps, const __half2* tab,
                         cudaStream_t stream) {
  using A = ApplyShape<R>;
  static bool done[64] = {false};
  const cudaError_t e = allow_smem(fma_tiled_apply<T, R, ROPE>, A::SMEM, done);
  if (e != cudaSuccess) return e;
  const long long tiles = (p.N + A::NT - 1) / A::NT;
  const int slots = sms() * A::CTAS;
  const long long few = (4ll * slots + p.units() - 1) / p.units();   // four waves: beyond that the last one is small anyway
  const int C = pieces(tiles, p.units(), slots, 1, tiles < few ? tiles : few, 0.3);
  fma_tiled_apply<T, R, ROPE><<<dim3(C, p.units()), A::THREADS, A::SMEM, stream>>>((const T*)q, state, (T*)o, p, eps, tab);
  count_launches(1);
  return cudaGetLastError();
}

#define LINATTN_TILED(FN, T, ROPE, ...)              \
  switch ((p.d + 15) / 16) {                         \
    case 1: return FN<T, 1, ROPE>(__VA_ARGS__);      \
    case 2: return FN<T, 2, ROPE>(__VA_ARGS__);      \
    case 3: return FN<T, 3, ROPE>(__VA_ARGS__);      \
    case 4: return FN<T, 4, ROPE>(__VA_ARGS__);      \
    case 5: return FN<T, 5, ROPE>(__VA_ARGS__);      \
    case 6: return FN<T, 6, ROPE>(__VA_ARGS__);      \
    case 7: return FN<T, 7, ROPE>(__VA_ARGS__);      \
    default: return FN<T, 8, ROPE>(__VA_ARGS__);     \
  }

}  // namespace

// The tiled kernels read rows in 16-byte pieces and the rotations of a piece in one load; everything else (odd head
// dims, unaligned views) takes the general kernels.
bool fma_tiled_ok(const Problem& p, const void* a, const void* b, const __half2* rope) {
  const int esz = p.dtype == LINATTN_F32 ? 4 : 2, per = 16 / esz;
  const uintptr_t tab_align = p.dtype == LINATTN_F32 ? 7 : 15;
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0 && p.d % per == 0 && p.sb % per == 0 &&
         p.sn % per == 0 && p.sh % per == 0 && (reinterpret_cast<uintptr_t>(rope) & tab_align) == 0;
}

cudaError_t fma_tiled_state_partials(const Problem& p, const void* k, const void* v, float* partials, const __half2* rope,
                                     int* P, cudaStream_t stream) {
  if (p.dtype == LINATTN_F32) {
    if (rope) { LINATTN_TILED(launch_state, float, true, p, k, v, partials, rope, P, stream) }
    LINATTN_TILED(launch_state, float, false, p, k, v, partials, rope, P, stream)
  }
  if (rope) { LINATTN_TILED(launch_state, __nv_bfloat16, true, p, k, v, partials, rope, P, stream) }
  LINATTN_TILED(launch_state, __nv_bfloat16, false, p, k, v, partials, rope, P, stream)
}

cudaError_t fma_tiled_apply_tokens(const Problem& p, const void* q, const float* state, void* o, float eps, const __half2* rope,
                                   cudaStream_t stream) {
  if (p.dtype == LINATTN_F32) {
    if (rope) { LINATTN_TILED(launch_apply, float, true, p, q, state, o, eps, rope, stream) }
    LINATTN_TILED(launch_apply, float, false, p, q, state, o, eps, rope, stream)
  }
  if (rope) { LINATTN_TILED(launch_apply, __nv_bfloat16, true, p, q, state, o, eps, rope, stream) }
  LINATTN_TILED(launch_apply, __nv_bfloat16, false, p, q, state, o, eps, rope, stream)
}

}  // namespace linattn
