// Included by umma_kernels.cu, whose helpers it uses.
//
// The state and apply passes with the CTAs of a unit as a thread-block cluster, for up to some thousand tokens.
//
// What the grid form (umma_fused_kernel) pays whatever the size is the way of the state from the accumulators to the apply
// operand: records to memory, a grid barrier, the reduce, a second barrier, the operand image back in (10 us), and a
// cooperative launch.  Here that way stays on chip.  Each of the c CTAs of a unit runs the state MMAs of its share of the
// tokens with a lane of the accumulators as a value feature (operands exchanged, as for lone CTAs), adds its tiles up in
// registers, and sends every row of the sums to the CTA that owns it, through distributed shared memory; the owners add the
// c sums (and the cache's state) in a fixed order, write the state out if somebody reads it, and send the row as bf16 hi + lo
// to the apply operand of all c CTAs.  What is sent goes in bulk copies, whose bytes arrive at a barrier of the CTA they go to:
// two such barriers take the place of the two grid barriers.  (Stores of 16 bytes a lane: 2300 cycles for the sums, 6200 for the
// operand; behind a fence of the cluster they took longer still.)
//
// A cluster has to fit into one GPC, so 148 SMs hold 15 to 74 clusters of eight to two CTAs, and with many tokens the grid, which
// uses all SMs, is faster: cluster_size draws the line.

// Addresses below are bytes behind the 1024-byte aligned start of shared memory.
template <int D, bool ROPE>
struct ClusterCfg {
  using C = Cfg<D>;
  static constexpr int MOST = 8;                                // CTAs of a cluster (the portable most)
  // Plain heads of 112: the ones that the ReLU role writes into value column 112 make lane 112 of the sums z, one more row.
  // Else z comes from the ReLU role's fp32 sums.
  static constexpr bool Z_LANE = D == 112 && !ROPE;
  static constexpr int ROWS = Z_LANE ? 113 : C::FEAT;
  static constexpr int ROW4 = D / 4;                            // float4 of a row: the columns of its own head
  static constexpr int CPR = D / 8;                             // chunks of eight columns of a row
  static constexpr int KOFF = 2 * kBox;                         // a stage: V0 V1 K0 K1 ...
  static constexpr int RECV_BYTES = (ROWS + MOST - 1) * D * 4;  // sums of the rows a CTA owns, from each CTA: c * ceil(ROWS / c) rows
  static constexpr int Z_BYTES = Z_LANE ? 0 : (kZSlots + MOST + 1) * 128 * 4;
  static constexpr int DEN_BYTES_OF(int slots) { return ROPE && D != 112 ? C::G * slots * kTileApply * 4 : 0; }
  static constexpr int LIMIT = 227 * 1024 - 1024 - C::BAR_BYTES;
  static constexpr int fit() {
    int n = 1;
    while (n < 5 && C::S_BYTES + (n + 1) * C::SLOT_BYTES + RECV_BYTES + Z_BYTES + DEN_BYTES_OF(n + 1) <= LIMIT) ++n;
    return n;
  }
  static constexpr int SLOTS = fit();
  static constexpr int RECV = C::S_BYTES + SLOTS * C::SLOT_BYTES;
  static constexpr int Z = (RECV + RECV_BYTES + 127) & ~127;    // [kZSlots][128] sums by warp, [MOST][128] by CTA, [128] z
  static constexpr int DEN = Z + Z_BYTES;
  static constexpr int BARS = (DEN + DEN_BYTES_OF(SLOTS) + 127) & ~127;
  // ... and, in the rotary variant, the rotations of its tokens, as in umma_fused_kernel, where three such stages fit (not at
  // d = 128: there the threads fetch them into registers).
  static constexpr bool TAB = ROPE && RECV / C::ROPE_STAGE_BYTES >= 3;
  static constexpr int STAGE = TAB ? C::ROPE_STAGE_BYTES : 4 * kBox;
  static constexpr int STAGES = RECV / STAGE < 4 ? RECV / STAGE : 4;
  static constexpr size_t SMEM = 1024 + BARS + C::BAR_BYTES;
  static_assert(SMEM <= 227 * 1024 && SMEM >= kSmemAlone && SLOTS >= 2, "shared memory of a cluster's CTA");
};

struct ClusterParams {
  int H, HG;               // HG: head groups per batch entry
  int tiles;               // 64-token tiles of a unit
  int c;                   // CTAs of a cluster
  int do_apply, accumulate, write_state;
  float* state;
  const float* state_base;
  float eps;
  WorkspaceCtrl* ctrl;
  const uint4* rope;
  long long N;
};

template <int D, bool ROPE>
__global__ void __launch_bounds__(Roles<ROPE>::THREADS, 1)
umma_cluster_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o,
                    const __grid_constant__ ClusterParams p) {
  using C = Cfg<D>;
  using L = ClusterCfg<D, ROPE>;
  using R = Roles<ROPE>;
  constexpr bool TAB = L::TAB;
  constexpr int TOFF = 4 * kBox;
  constexpr int NSA = L::STAGES, NSC = L::SLOTS, STAGE = L::STAGE, KOFF = L::KOFF, SLOT = C::SLOT_BYTES, HALF = SLOT / 2;
  constexpr uint32_t IDESC_A = make_idesc_bf16(128, C::FEAT, true, true);
  constexpr uint32_t IDESC_C = make_idesc_bf16(128, C::NAPPLY, false, false);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* s_op = smem;                    // apply operand ...
  uint8_t* slots = smem + C::S_BYTES;      // ... and Q/O slots; the state pass stages lie over both
  float* recv = reinterpret_cast<float*>(smem + L::RECV);   // [c][ROW4][rows]: float4
  float* z_slots = reinterpret_cast<float*>(smem + L::Z);
  float* z_recv = z_slots + kZSlots * 128;
  float* z_row = z_recv + L::MOST * 128;
  float* den_rows = reinterpret_cast<float*>(smem + L::DEN);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::BARS);
  uint64_t* a_full = bars;                 // state pass, as in umma_fused_kernel
  uint64_t* a_ready = a_full + NSA;
  uint64_t* a_empty = a_ready + NSA;
  uint64_t* a_tfull = a_empty + NSA;       // [2] the tile's accumulators are complete
  uint64_t* a_tempty = a_tfull + 2;        // [2] ... and read
  uint64_t* a_done = a_tempty + 2;         // every MMA of the state pass is complete
  uint64_t* z_left = a_done + 1;           // the warps' sums for z are in shared memory
  uint64_t* x_full = z_left + 1;           // every CTA's sums of this CTA's rows have come
  uint64_t* s_full = x_full + 1;           // the apply operand is complete
  uint64_t* x_staged = s_full + 1;         // the sums for the peers are in shared memory
  uint64_t* s_staged = x_staged + 1;       // ... and this CTA's rows of the operand
  uint64_t* c_full = s_staged + 1;         // apply pass, as in umma_fused_kernel
  uint64_t* c_ready = c_full + NSC;
  uint64_t* c_empty = c_ready + NSC;
  uint64_t* c_staged = c_empty + NSC;
  uint64_t* c_tfull = c_staged + NSC;      // [2]
  uint64_t* c_tempty = c_tfull + 2;        // [2]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(c_tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  static_assert((3 * NSA + 10 + 4 * NSC + 4) * 8 + 8 <= C::BAR_BYTES, "barrier block too small");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = p.c, rank = (int)cluster_rank(), u = (int)blockIdx.x / c, b = u / p.HG, hg = u % p.HG;
  // this CTA's share of the unit: 64-token tiles [t0, t0 + n), in the apply pass two to a tile of 128 rows
  const int t0 = (int)((long long)p.tiles * rank / c), n = (int)((long long)p.tiles * (rank + 1) / c) - t0;
  const int n_apply = p.do_apply ? (n + 1) / 2 : 0;
  const int rows = (L::ROWS + c - 1) / c;   // rows a CTA owns: [rank * rows, + rows_here)
  const int rows_here = L::ROWS - rank * rows < rows ? L::ROWS - rank * rows : rows;
  constexpr int OWN_THREADS = R::RELU_THREADS + 128, OWN_WARPS = OWN_THREADS / 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSA; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_ready[s], R::RELU_THREADS + (ROPE ? 128 : 0)); mbar_init(&a_empty[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&a_tfull[i], 1); mbar_init(&a_tempty[i], 128); mbar_init(&c_tfull[i], 1); mbar_init(&c_tempty[i], 128); }
    mbar_init(a_done, 1);
    mbar_init(z_left, R::RELU_THREADS + (ROPE ? 128 : 0));
    mbar_init(x_full, 1 + 4);
    mbar_init(x_staged, 4);
    mbar_init(s_staged, OWN_WARPS);
    mbar_init(s_full, 1 + OWN_WARPS);
    for (int s = 0; s < NSC; ++s) {
      mbar_init(&c_full[s], 1); mbar_init(&c_ready[s], R::RELU_THREADS); mbar_init(&c_empty[s], 1); mbar_init(&c_staged[s], 128);
    }
    mbar_arrive_expect_tx(x_full, ((c - 1) * rows_here * D + (L::Z_LANE ? 0 : c * 128)) * 4);
    mbar_arrive_expect_tx(s_full, (L::ROWS - rows_here) * 4 * kRowBytes);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tensormap(&map_k);
    prefetch_tensormap(&map_v);
  }
  wait_for_prior_grids();
  if (warp == 1) { tmem_alloc(tmem_holder, kTmemCols); tmem_relinquish(); }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  let_next_grid_start();
  const uint32_t tmem_base = *tmem_holder;
  cluster_arrive();   // the peers' barriers are set up: waited for before the first access to a peer

  // ---- Q tiles: two boxes of 64 tokens each per 64-feature box; the second half of a last odd tile is not loaded (its rows
  // hold what was there before; rows do not mix, and they are not stored)
  int c_it = 0;
  auto load_q_tile = [&]() -> bool {
    const int s = c_it % NSC, halves = 2 * c_it + 1 < n ? 2 : 1;
    if (!mbar_wait(&c_empty[s], ((c_it / NSC) & 1) ^ 1, abort_flag)) return false;
    uint8_t* sl = slots + s * SLOT;
    mbar_arrive_expect_tx(&c_full[s], halves * 2 * kBox);
    for (int h = 0; h < halves; ++h)
      for (int box = 0; box < 2; ++box) {
        int c0, c1;
        box_coords<D>(box, hg, c0, c1);
        tma_load_4d(sl + box * HALF + h * kBox, &map_q, &c_full[s], c0, c1, (t0 + 2 * c_it + h) * kTileState, b);
      }
    ++c_it;
    return true;
  };

  // ---- what both the state pass and the exchange behind it need
  const int tr = threadIdx.x - kReluThread0;                       // ReLU role
  const int row0 = tr >> 3, pc = tr & 7, lc = pc ^ (row0 & 7);     // its rows, and the 16-byte chunk it holds of all of them
  const bool box1_live = 64 + lc * 8 < C::FEAT;
  // z: one thread a feature, in every CTA.  A step writes the new z where the old one is, and the CTAs of a cluster go at their
  // own pace: the old z is read by the threads that write the new one (rank 0's), and before they send theirs, so that what they
  // write behind everybody's sums nobody reads.
  const int zh = hg * C::G + tr / D;
  const bool z_owned = !L::Z_LANE && rank == 0 && (unsigned)tr < (unsigned)C::FEAT && zh < p.H;   // (a head there is, not padding of the group)
  auto z_at = [&] { return ((size_t)(b * p.H + hg * C::G + tr / D) * (D + 1) + D) * D + tr % D; };

  // ==================================================================== state pass
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      for (int it = 0; it < n; ++it) {
        const int s = it % NSA;
        if (!mbar_wait(&a_empty[s], ((it / NSA) & 1) ^ 1, abort_flag)) break;
        uint8_t* st = smem + s * STAGE;
        if (TAB) {
          const long long m = (long long)(t0 + it) * kTileState, left = p.N - m;
          const uint32_t bytes = (left < kTileState ? (uint32_t)left : (uint32_t)kTileState) * C::TAB_ROW;
          mbar_arrive_expect_tx(&a_full[s], 4 * kBox + bytes);
          bulk_load(st + TOFF, p.rope + m * (D / 8), bytes, &a_full[s]);
        } else {
          mbar_arrive_expect_tx(&a_full[s], 4 * kBox);
        }
        for (int box = 0; box < 2; ++box) {
          int c0, c1;
          box_coords<D>(box, hg, c0, c1);
          tma_load_4d(st + KOFF + box * kBox, &map_k, &a_full[s], c0, c1, (t0 + it) * kTileState, b);
          tma_load_4d(st + box * kBox, &map_v, &a_full[s], c0, c1, (t0 + it) * kTileState, b);
        }
      }
      // Q does not depend on the state: its first tiles as soon as the stages are free
      if (n_apply > 0 && mbar_wait(a_done, 0, abort_flag))
        while (c_it < n_apply && c_it < NSC)
          if (!load_q_tile()) break;
    }
    cluster_wait();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int it = 0;
      for (; it < n; ++it) {
        const int s = it % NSA, set = it & 1;
        // Plain: two accumulators collect a tile's four K steps while the other two are read, so no chain of the tensor
        // core's truncating additions is longer than two (a lone tile has all four: one).  Rotary: the accumulators are read
        // once, behind the last tile; each takes one K step of every tile, so a chain is as long as the CTA has tiles.  (Whole
        // tiles in turn made chains of four times a quarter of that, rounded up.  2-norm of S against 64 bits with factors that
        // turn nothing, whole tiles / K steps / the forms without clusters: 192 tokens, 3 heads of 64 5.54e-8 / 4.72e-8 / 4.72e-8;
        // 1200 tokens, 4 heads of 112 7.71e-8 / 7.38e-8 / 9.03e-8; 4680 tokens, 20 heads 1.305e-7 / 1.303e-7 / 1.209e-7.  Turned
        // keys are rounded to bf16: 1.6e-3 in all of them.)
        if (!ROPE && it >= 2 && !mbar_wait(&a_tempty[set], ((it - 2) >> 1) & 1, abort_flag)) break;
        if (!mbar_wait(&a_ready[s], (it / NSA) & 1, abort_flag)) break;
        tcgen05_fence_after();
        const uint32_t st = smem_u32(smem + s * STAGE);
#pragma unroll
        for (int kk = 0; kk < kTileState / 16; ++kk) {
          const uint64_t kd = make_smem_desc_sw128(st + KOFF + kk * 2048, kBox, 1024);   // phi(K), MN-major
          const uint64_t vd = make_smem_desc_sw128(st + kk * 2048, kBox, 1024);          // V^T, MN-major
          const int acc = ROPE || n == 1 ? kk : 2 * set + (kk & 1);
          const bool first = ROPE ? it == 0 : n == 1 || kk < 2;
          umma_bf16(tmem_base + acc * 128, vd, kd, IDESC_A, first ? 0u : 1u);
        }
        umma_commit(&a_empty[s]);
        if (!ROPE) umma_commit(&a_tfull[set]);
      }
      if (it > 0) umma_commit(a_done); else mbar_arrive(a_done);
    }
    cluster_wait();
  } else if (warp < R::EPI_WARP0) {
    // ------------------------------------------------------------ ReLU pass over the K boxes
    float2 zacc[8];   // sums of the plain phi(k): features 8 * lc.. of box 0, 64 + 8 * lc.. of box 1
#pragma unroll
    for (int e = 0; e < 8; ++e) zacc[e] = make_float2(0.f, 0.f);
    // rotary variant: this role takes box 0 and half the rows of box 1, the epilogue the other half; rotations one tile ahead
    uint4 tab0[kTileState / 32], tab1;
    const uint4* const rope = ROPE && !TAB ? behind_wait(p.rope) : nullptr;
    auto fetch_rot = [&](int tile, int i) {
      const long long m = (long long)tile * kTileState + row0 + 32 * i;
      tab0[i] = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
      if (i == 0) tab1 = tab0[i];
      if (m < p.N) {
        tab0[i] = __ldg(rope + m * (D / 8) + C::tab_chunk(0, lc));
        if (i == 0) {
          if (C::SAME_TAB) tab1 = tab0[0];
          else if (box1_live) tab1 = __ldg(rope + m * (D / 8) + C::tab_chunk(1, lc));
        }
      }
    };
    if (ROPE && !TAB) {
#pragma unroll
      for (int i = 0; i < kTileState / 32; ++i) fetch_rot(t0, i);
    }
    bool ok = true;
    for (int it = 0; it < n && ok; ++it) {
      const int s = it % NSA;
      uint8_t* st = smem + s * STAGE;
      ok = __all_sync(0xffffffffu, mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag));
      if (!ok) break;
      if (TAB) {
        rope_state_rows<D>(st + KOFF, st + TOFF, row0, pc, lc, p.N - (long long)(t0 + it) * kTileState - row0, zacc);
      } else if (ROPE) {
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
            *c1 = rotate_pack8(f, tab1);
          }
          if (it + 1 < n) fetch_rot(t0 + it + 1, i);
        }
      } else if (L::Z_LANE) {
        relu_pass<C::FEAT, kTileState>(st + KOFF, st + KOFF + kBox, tr);
        // value column 112 := 1 (logical chunk 6 of the second V box, element 0): lane 112 of the sums is z
        if (tr < kTileState) *reinterpret_cast<uint16_t*>(st + kBox + tr * kRowBytes + ((6 ^ (tr & 7)) << 4)) = 0x3F80u;
      } else {
        relu_sum_pass<C::FEAT, kTileState>(st + KOFF, st + KOFF + kBox, tr, zacc);
      }
      fence_proxy_async_smem();
      mbar_arrive(&a_ready[s]);
    }
    if (C::G > 1 && p.do_apply) {   // blocks across heads are zero; the others are stored below, but not before z has come from here
      ok = ok && __all_sync(0xffffffffu, mbar_wait(a_done, 0, abort_flag));
      if (ok) {
        for (int i = tr; i < 4 * rows_here * (kRowBytes / 16); i += R::RELU_THREADS) {   // (this CTA's rows: the peers send whole ones)
          const int block = i / (rows_here * (kRowBytes / 16)), at = i - block * (rows_here * (kRowBytes / 16));
          *reinterpret_cast<uint4*>(s_op + block * C::SBOX_BYTES + rank * rows * kRowBytes + at * 16) = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async_smem();
      }
    }
    const float z_old = z_owned && p.accumulate ? __ldcg(behind_wait(p.state_base) + z_at()) : 0.f;
    if (!L::Z_LANE && ok) {
      leave_z(z_slots, zacc, tr, lc, box1_live);
      mbar_arrive(z_left);
      ok = mbar_wait(z_left, 0, abort_flag);
    }
    cluster_wait();
    if (!L::Z_LANE && ok && tr < 128) {
      const float z = z_old + (tr < C::FEAT ? sum_z_slots<ROPE>(z_slots, tr) : 0.f);
      for (int r = 0; r < c; ++r) store_async(cluster_address(z_recv + rank * 128 + tr, r), cluster_address(x_full, r), z);
    }
  } else if (warp < R::STORE_WARP) {
    // ------------------------------------------------------------ epilogue: the tiles' sums, then each row to its owner
    const int wq = warp & 3, j = wq * 32 + lane;          // accumulator lane = value feature within the group
    const int g0 = C::G == 1 ? 0 : wq * 32 / D;           // its head (one to a warp)
    const uint32_t trow = tmem_base + ((uint32_t)(wq * 32) << 16) + g0 * D;   // the columns of that head
    const int te = threadIdx.x - R::EPI_THREAD0;
    bool ok = true;
    float sum[D];
    if (ROPE) {
      // token rows 32..63 of the second K box of every tile (see the ReLU role)
      const int row0h = te >> 3, pch = te & 7, lch = pch ^ (row0h & 7);
      const bool h_live = 64 + lch * 8 < C::FEAT;
      float2 zh[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) zh[e] = make_float2(0.f, 0.f);
      uint4 tabh[2];
      const uint4* const rope = ROPE && !TAB ? behind_wait(p.rope) : nullptr;
      auto fetch_roth = [&](int tile, int i) {
        const long long m = (long long)tile * kTileState + 32 + row0h + 16 * i;
        tabh[i] = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
        if (h_live && m < p.N) tabh[i] = __ldg(rope + m * (D / 8) + C::tab_chunk(1, lch));
      };
      if (!TAB) {
        fetch_roth(t0, 0);
        fetch_roth(t0, 1);
      }
      for (int it = 0; it < n; ++it) {
        const int s = it % NSA;
        ok = __all_sync(0xffffffffu, mbar_wait(&a_full[s], (it / NSA) & 1, abort_flag));
        if (!ok) break;
        uint8_t* p1 = smem + s * STAGE + KOFF + kBox + (32 + row0h) * kRowBytes + pch * 16;
        if (TAB) {
          const uint8_t* tb = smem + s * STAGE + TOFF + (32 + row0h) * C::TAB_ROW + C::tab_chunk(1, lch) * 16;
          const long long rows_left = p.N - (long long)(t0 + it) * kTileState - 32 - row0h;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            tabh[i] = make_uint4(kRopeIdentity, kRopeIdentity, kRopeIdentity, kRopeIdentity);
            if (h_live && rows_left > 16 * i) tabh[i] = *reinterpret_cast<const uint4*>(tb + i * 16 * C::TAB_ROW);
          }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (h_live) {
            float2 f[4];
            uint4* c1 = reinterpret_cast<uint4*>(p1 + i * 16 * kRowBytes);
            unpack_relu8(*c1, f);
#pragma unroll
            for (int e = 0; e < 4; ++e) zh[e] = add2(zh[e], f[e]);
            *c1 = rotate_pack8(f, tabh[i]);
          }
          if (!TAB && it + 1 < n) fetch_roth(t0 + it + 1, i);
        }
        fence_proxy_async_smem();
        mbar_arrive(&a_ready[s]);
      }
      if (ok) {   // this warp's share of z: the four lanes that share a chunk add up in a fixed order
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
          float* zp = z_slots + (8 + (te >> 5)) * 128 + 64 + 8 * lch;
          *reinterpret_cast<float4*>(zp) = make_float4(tot[0], tot[1], tot[2], tot[3]);
          *reinterpret_cast<float4*>(zp + 4) = make_float4(tot[4], tot[5], tot[6], tot[7]);
        }
        mbar_arrive(z_left);
      }
      ok = ok && __all_sync(0xffffffffu, mbar_wait(a_done, 0, abort_flag));
      if (ok) tcgen05_fence_after();
    }
    cluster_wait();
    // Rows to their owners, [rank][float4 of the row][row] there, so that neighbouring lanes write neighbouring 16 bytes; on
    // the way they wait where the owner's rows of the operand will come in (eight float4 of a row in the 128 bytes of a block of
    // four), which the owner sends only when it has them.
    const int owner = j / rows, jl = j - owner * rows, owned = L::ROWS - owner * rows < rows ? L::ROWS - owner * rows : rows;
    float4* const own_at = reinterpret_cast<float4*>(recv) + rank * L::ROW4 * rows_here + jl;
    uint8_t* const away_at = s_op + owner * rows * kRowBytes + jl * 16;
    auto put = [&](int k, const float4& x) {
      if (owner == rank) own_at[k * rows_here] = x;
      else *reinterpret_cast<float4*>(away_at + (k >> 3) * C::SBOX_BYTES + (k & 7) * owned * 16) = x;
    };
    if (ROPE) {
      if (ok) {
#pragma unroll 1
        for (int cc = 0; cc < D / 16; ++cc) {
          float v[16];
          uint32_t r[4][16];
#pragma unroll
          for (int a = 0; a < 4; ++a) tmem_ld_x16(trow + a * 128 + cc * 16, r[a]);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 16; ++x)
            v[x] = ((__uint_as_float(r[0][x]) + __uint_as_float(r[1][x])) + __uint_as_float(r[2][x])) + __uint_as_float(r[3][x]);
          if (j < L::ROWS) {
#pragma unroll
            for (int k = 0; k < 4; ++k) put(cc * 4 + k, make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]));
          }
        }
      }
    } else {
      for (int it = 0; it < n; ++it) {
        const int set = it & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&a_tfull[set], (it >> 1) & 1, abort_flag));
        if (!ok) break;
        tcgen05_fence_after();
#pragma unroll
        for (int cc = 0; cc < D / 16; ++cc) {
          uint32_t r[2][16];
          tmem_ld_x16(trow + (2 * set) * 128 + cc * 16, r[0]);
          tmem_ld_x16(trow + (2 * set + 1) * 128 + cc * 16, r[1]);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 16; ++x) {
            const float two = __uint_as_float(r[0][x]) + __uint_as_float(r[1][x]);
            sum[cc * 16 + x] = it == 0 ? two : sum[cc * 16 + x] + two;
          }
          if (n == 1) {
            tmem_ld_x16(trow + 2 * 128 + cc * 16, r[0]);
            tmem_ld_x16(trow + 3 * 128 + cc * 16, r[1]);
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 16; ++x) sum[cc * 16 + x] = (sum[cc * 16 + x] + __uint_as_float(r[0][x])) + __uint_as_float(r[1][x]);
          }
        }
        tcgen05_fence_before();
        mbar_arrive(&a_tempty[set]);
      }
      if (ok && j < L::ROWS) {
#pragma unroll
        for (int k = 0; k < L::ROW4; ++k) put(k, make_float4(sum[4 * k], sum[4 * k + 1], sum[4 * k + 2], sum[4 * k + 3]));
      }
    }
    tcgen05_fence_before();
    if (ok) {
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) { mbar_arrive(x_full); mbar_arrive(x_staged); }
      if (warp == R::EPI_WARP0 && __all_sync(0xffffffffu, mbar_wait(x_staged, 0, abort_flag))) {
        constexpr int BLOCKS = (L::ROW4 + 7) / 8;   // of eight float4 of a row
        for (int i = lane; i < (c - 1) * BLOCKS; i += 32) {
          const int peer = i / BLOCKS + (i / BLOCKS >= rank ? 1 : 0), block = i % BLOCKS;
          const int theirs = L::ROWS - peer * rows < rows ? L::ROWS - peer * rows : rows, wide = L::ROW4 - 8 * block < 8 ? L::ROW4 - 8 * block : 8;
          bulk_copy_cluster(cluster_address(reinterpret_cast<float4*>(recv) + (rank * L::ROW4 + 8 * block) * theirs, peer),
                            s_op + block * C::SBOX_BYTES + peer * rows * kRowBytes, wide * theirs * 16, cluster_address(x_full, peer));
        }
      }
    }
  } else {
    cluster_wait();
  }

  int q_done = 0;   // Q tiles that this warp of the ReLU role has clamped before the apply pass

  // ==================================================================== the rows this CTA owns: sum, state, apply operand
  if (warp >= 2 && warp < R::STORE_WARP) {
    constexpr int ITEMS = ((L::ROWS + 1) / 2 * L::CPR + OWN_THREADS - 1) / OWN_THREADS;   // of a thread, with two CTAs or more
    const int ot = tr;
    float4 acc[ITEMS][2];
    int j_of[ITEMS], q_of[ITEMS];
    size_t at_of[ITEMS];
    const float* const base = behind_wait(p.state_base);
    const int recip = ((1 << 20) + rows_here - 1) / rows_here;
    static_assert(ITEMS * OWN_THREADS * 64 < 1 << 20, "recip");
    bool live[ITEMS], held[ITEMS];   // held: a head there is, not padding of the group
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {   // the old state is asked for before the wait
      const int idx = ot + k * OWN_THREADS, q = (idx * recip) >> 20, j = rank * rows + (idx - q * rows_here);   // (idx / rows_here)
      live[k] = q < L::CPR;
      const int g = C::G == 1 ? 0 : j / D, il = j - g * D, h = hg * C::G + g;
      held[k] = live[k] && h < p.H;
      j_of[k] = j; q_of[k] = q;
      at_of[k] = ((size_t)(b * p.H + h) * (D + 1) + il) * D + q * 8;
      acc[k][0] = acc[k][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p.accumulate && held[k]) {
        acc[k][0] = __ldcg(reinterpret_cast<const float4*>(base + at_of[k]));
        acc[k][1] = __ldcg(reinterpret_cast<const float4*>(base + at_of[k]) + 1);
      }
    }

    // Plain: the Q tiles that have come are clamped while the peers' sums and the old state are on their way, not behind the operand: 900 cycles
    // of the 18 000 that a forward of 192 tokens, 4 heads of 32 takes.  (The old state is asked for first.  Behind the clamping its way began when
    // the sums had come, and the operand waited for it.  Steps, us, behind / first: 500 tokens, 56 heads of 112 18.9 / 16.5, 2300 tokens,
    // 40 heads 29.0 / 27.2, 300 tokens, 4 heads 11.9 / 11.6, 150 tokens, 18 heads of 128 14.5 / 14.2; but 700 tokens, 20 heads 14.2 / 14.4.)
    if (!ROPE && warp < R::EPI_WARP0) {
      const int most = n_apply < NSC ? n_apply : NSC;
      for (int spin = 0; spin < 4096 && q_done < most && !__all_sync(0xffffffffu, mbar_test(x_full, 0)); ++spin) {
        if (!__all_sync(0xffffffffu, mbar_test(&c_full[q_done], 0))) continue;
        relu_pass<C::FEAT, kTileApply>(slots + q_done * SLOT, slots + q_done * SLOT + HALF, tr);
        fence_proxy_async_smem();
        mbar_arrive(&c_ready[q_done]);
        ++q_done;
      }
    }

    if (__all_sync(0xffffffffu, mbar_wait_cluster(x_full, 0, abort_flag))) {
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) {
        if (!live[k]) continue;
        const float4* src = reinterpret_cast<const float4*>(recv) + (2 * q_of[k]) * rows_here + (j_of[k] - rank * rows);
        for (int r = 0; r < c; ++r) {
          add4(acc[k][0], src[r * L::ROW4 * rows_here]);
          add4(acc[k][1], src[r * L::ROW4 * rows_here + rows_here]);
        }
        if (p.write_state && held[k]) {
          reinterpret_cast<float4*>(p.state + at_of[k])[0] = acc[k][0];
          reinterpret_cast<float4*>(p.state + at_of[k])[1] = acc[k][1];
        }
        if (p.do_apply) {
          const float x8[8] = {acc[k][0].x, acc[k][0].y, acc[k][0].z, acc[k][0].w, acc[k][1].x, acc[k][1].y, acc[k][1].z, acc[k][1].w};
          uint4 hi, lo;
          split_hi_lo(x8, hi, lo);
          const int i0 = (C::G == 1 ? 0 : j_of[k] / D * D) + q_of[k] * 8;   // first key feature of the chunk
          uint8_t* to = s_op + (i0 >> 6) * C::SBOX_BYTES + j_of[k] * kRowBytes + ((((i0 & 63) >> 3) ^ (j_of[k] & 7)) << 4);
          *reinterpret_cast<uint4*>(to) = hi;
          *reinterpret_cast<uint4*>(to + 2 * C::SBOX_BYTES) = lo;
        }
      }
      if (!L::Z_LANE && ot < C::FEAT) {
        float z = 0.f;
        for (int r = 0; r < c; ++r) z += z_recv[r * 128 + ot];   // (rank 0's has the old z in it)
        if (z_owned && p.write_state) p.state[z_at()] = z;
        if (ROPE) z_row[ot] = z;
        else if (p.do_apply) put_z<D>(s_op, ot, z);
      }
      fence_proxy_async_smem();   // the rows are copied, and read by the MMAs
      __syncwarp();
      if (lane == 0) { mbar_arrive(s_full); mbar_arrive(s_staged); }
      if (p.do_apply && warp == 2 && __all_sync(0xffffffffu, mbar_wait(s_staged, 0, abort_flag))) {
        for (int i = lane; i < (c - 1) * 4; i += 32) {   // this CTA's rows of the four blocks to every peer
          const int peer = i / 4 + (i / 4 >= rank ? 1 : 0);
          uint8_t* at = s_op + (i & 3) * C::SBOX_BYTES + rank * rows * kRowBytes;
          bulk_copy_cluster(cluster_address(at, peer), at, rows_here * kRowBytes, cluster_address(s_full, peer));
        }
      }
    }
  }
  // No CTA leaves before all have what was sent to them: every warp says so as soon as it knows (those above have seen the sums come and
  // have sent the operand, the MMA warp sees the operand complete; the other two send and get nothing), and the end of the
  // kernel only looks; said and waited for there, it took 2000 cycles.  With both, before and after, us: read-only rotary step of 4680 tokens
  // 35.85 -> 35.10, rotary forward of 1625 tokens, 20 heads of 112 20.5 -> 19.7, plain steps of 431 14.3 -> 13.9, of 713 14.65 -> 14.14.
  bool operand = n_apply == 0;
  if (warp == 1 && n_apply > 0) operand = __all_sync(0xffffffffu, mbar_wait_cluster(s_full, 0, abort_flag));
  __syncwarp();
  cluster_arrive();

  // ==================================================================== apply pass
  if (warp == 0) {
    if (lane == 0) {
      while (c_it < n_apply)
        if (!load_q_tile()) break;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0 && n_apply > 0) {
      bool ok = operand;
      fence_proxy_async_smem();
      for (int it = 0; it < n_apply && ok; ++it) {
        const int s = it % NSC, acc = it & 1;
        ok = mbar_wait(&c_tempty[acc], ((it >> 1) & 1) ^ 1, abort_flag) && mbar_wait(&c_ready[s], (it / NSC) & 1, abort_flag);
        if (!ok) break;
        tcgen05_fence_after();
        const uint32_t a0 = smem_u32(slots + s * SLOT), b0 = smem_u32(s_op);
#pragma unroll
        for (int k = 0; k < C::KSTEPS; ++k) {
          const uint32_t boff = (k >> 2) * C::SBOX_BYTES + (k & 3) * 32;
          const uint64_t a = make_smem_desc_sw128(a0 + (k >> 2) * HALF + (k & 3) * 32, 16, 1024);   // phi(Q), K-major
          const uint64_t bh = make_smem_desc_sw128(b0 + boff, 16, 1024);                            // S hi
          const uint64_t bl = make_smem_desc_sw128(b0 + 2 * C::SBOX_BYTES + boff, 16, 1024);        // S lo
          umma_bf16(tmem_base + acc * kAccStride, a, bh, IDESC_C, k == 0 ? 0u : 1u);
          umma_bf16(tmem_base + acc * kAccStride, a, bl, IDESC_C, 1u);
        }
        umma_commit(&c_tfull[acc]);
      }
    }
  } else if (warp < R::EPI_WARP0) {
    // ------------------------------------------------------------ ReLU pass over the Q tiles
    float2 zc[8];   // rotary variant: z at this thread's features
    uint4 tab0[kTileApply / 32], tab1[kTileApply / 32];
#pragma unroll
    for (int i = 0; i < kTileApply / 32; ++i) tab0[i] = tab1[i] = make_uint4(0, 0, 0, 0);
    auto fetch_rot = [&](int it, int i) {   // (as in umma_fused_kernel)
      const long long x = (long long)(t0 + 2 * it) * kTileState + row0 + 32 * i;
      const uint4* at = p.rope + x * (D / 8);
      load_in_place(tab0[i], at + C::tab_chunk(0, lc), x < p.N);
      if (!C::SAME_TAB) load_in_place(tab1[i], at + C::tab_chunk(1, lc), x < p.N);
    };
    bool ok = true;
    if (ROPE && n_apply > 0) {
#pragma unroll
      for (int i = 0; i < kTileApply / 32; ++i) fetch_rot(0, i);
      // z_row is this CTA's own work: it is there with its rows of the operand, before the peers' have come
      ok = __all_sync(0xffffffffu, mbar_wait(s_staged, 0, abort_flag));
#pragma unroll
      for (int box = 0; box < 2; ++box) {
        float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
        if (ok && (box == 0 || box1_live)) {
          a0 = *reinterpret_cast<const float4*>(z_row + 64 * box + 8 * lc);
          a1 = *reinterpret_cast<const float4*>(z_row + 64 * box + 8 * lc + 4);
        }
        zc[4 * box + 0] = make_float2(a0.x, a0.y); zc[4 * box + 1] = make_float2(a0.z, a0.w);
        zc[4 * box + 2] = make_float2(a1.x, a1.y); zc[4 * box + 3] = make_float2(a1.z, a1.w);
      }
    }
    for (int it = q_done; it < n_apply && ok; ++it) {
      const int s = it % NSC;
      uint8_t* sl = slots + s * SLOT;
      ok = __all_sync(0xffffffffu, mbar_wait(&c_full[s], (it / NSC) & 1, abort_flag));
      if (!ok) break;
      if (ROPE) rope_apply_rows<D>(sl, den_rows + s * C::G * kTileApply, row0, pc, lc, zc, tab0, tab1, [&](int i) {
        fetch_rot(it + 1 < n_apply ? it + 1 : it, i);
      });
      else relu_pass<C::FEAT, kTileApply>(sl, sl + HALF, tr);
      fence_proxy_async_smem();
      mbar_arrive(&c_ready[s]);
    }
  } else if (warp < R::STORE_WARP) {
    // ------------------------------------------------------------ epilogue: divide, round, stage the O tile
    for (int it = 0; it < n_apply; ++it) {
      const int s = it % NSC, acc = it & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&c_tfull[acc], (it >> 1) & 1, abort_flag))) break;
      tcgen05_fence_after();
      apply_epilogue<D, ROPE>(tmem_base, acc, slots, s, den_rows, warp & 3, (warp & 3) * 32 + lane, p.eps, c_tempty);
      fence_proxy_async_smem();
      mbar_arrive(&c_staged[s]);
    }
  } else if (lane == 0) {
    // ------------------------------------------------------------ store warp: O tiles out, slots back to the producer
    constexpr bool kKeepStores = (C::FEAT * 2) % 128 != 0;   // (see umma_fused_kernel)
    const uint64_t policy = kKeepStores ? make_l2_policy_evict_last() : 0;
    for (int it = 0; it < n_apply; ++it) {
      const int s = it % NSC, halves = 2 * it + 1 < n ? 2 : 1;
      if (!mbar_wait(&c_staged[s], (it / NSC) & 1, abort_flag)) break;
      uint8_t* sl = slots + s * SLOT;
      for (int h = 0; h < halves; ++h)
        for (int box = 0; box < 2; ++box) {
          int c0, c1;
          box_coords<D>(box, hg, c0, c1);
          const int tok = (t0 + 2 * it + h) * kTileState;
          if (kKeepStores) tma_store_4d_hint(&map_o, sl + box * HALF + h * kBox, c0, c1, tok, b, policy);
          else tma_store_4d(&map_o, sl + box * HALF + h * kBox, c0, c1, tok, b);
        }
      tma_store_commit();
      tma_store_wait_read();
      mbar_arrive(&c_empty[s]);
    }
    tma_store_wait_all();
  }

  // ------------------------------------------------------------ teardown
  tcgen05_fence_before();
  __syncthreads();
  cluster_wait();   // nobody leaves while a peer may still write here (whatever is written has been sent by now)
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      p.ctrl->status = LINATTN_ERR_TIMEOUT;
      // what is still in flight targets this CTA's shared memory: give each stage, and what the peers send, a bounded wait
      for (int s = 0; s < NSA + NSC + 2; ++s)
        for (int par = 0; par < 2; ++par)
          for (int spin = 0; spin < 4096 && !mbar_try_wait(s < NSA ? &a_full[s] : s < NSA + NSC ? &c_full[s - NSA] : s == NSA + NSC ? x_full : s_full, par); ++spin)
            __nanosleep(64);
    }
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}
