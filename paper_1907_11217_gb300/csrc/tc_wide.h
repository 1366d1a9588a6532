// Wide-tile split-precision product (part of k_gemm_tc.cu: included inside
// its anonymous namespace, after the PTX helpers). Products with more than
// 64 complex columns; in BF16 and TF32 those for which wide_pays() says so.
//
// Tiles of 128 rows by 128 complex columns. Instead of one real product on
// the interleaved view, the complex product is formed from its planes, four
// real products per split term into two accumulators of 128 columns:
//     D_re += A_re B_re - A_im B_im       D_im += A_re B_im + A_im B_re
// (the minus sign is the instruction descriptor's negate-A bit). B is then
// stored once per value instead of twice (the interleaved view holds every
// component of B in two rows), and each byte of A and B feeds twice the
// products: a k-block of 64 real K brings 32 KB of A and 32 KB of B into the
// SM for 24 products of 64 cycles (42.7 B per cycle), where the interleaved
// form brings the same 64 KB for 12 (85 B per cycle, above what an SM's L2
// port sustains). The split arithmetic, barrier hand-overs and commits of a
// k-block are also spread over twice the tensor work.
//
// The accumulators form a ring of half-ranges (D_re, D_im, D_re, ...). A drain
// takes about 2000 cycles from the last product to the next product into the
// same columns (commit, the epilogue's wake-up, its loads beside the products'
// own accumulator traffic, hand-over), so it has to overlap the products of
// another half-range. BF16 and TF32 multiply two k-blocks into D_re, then the
// same two into D_im, in a ring of two. FP16, whose split warps deliver a
// k-block just in time, alternates per k-block and has a third accumulator,
// with two A slots instead of three (M16384 N1024 K2048 529 -> 507 us).
// A and B stages are separate rings: the split warps free an A stage as soon
// as they have read it, while a B stage lives until its products retire.
//
// Warps (four warpgroups; registers reassigned with setmaxnreg, 40 + 120 +
// 176 + 176 = 4 x 128, the launch's own total):
//   0 A loads, 1 MMA issuer, 2 readiness waiter, 3 B loads;
//   4..7  split A (one row of the tile a thread) into re / im, hi / lo;
//   8..15 epilogue: 64 complex columns of a row a thread, in registers.

// K (complex values) per k-block: a row of A is 32 floats (TF32) or 64.
template <int MODE>
__host__ __device__ constexpr int wide_kc() { return MODE == MODE_TF32 ? 16 : 32; }

constexpr int kWideCols = 128;  // complex columns per tile
// CG = 2: clusters of two CTAs on tiles of 256 rows (cta_group::2 products
// issued by the first CTA): each CTA loads and splits its own 128 rows of A and
// loads half of B, and drains its own rows of the accumulators. The pair
// signals across the cluster as in tc_split3_kernel.
constexpr int kWideThreads = 512;
constexpr unsigned long long kPairNs = 60000000000ull;  // 60 s
template <int MODE, int CG>
constexpr int kWideGroup = MODE == MODE_F16 ? 1 : 2;
// accumulators in the ring
template <int MODE, int CG>
constexpr int kWideAcc = MODE == MODE_F16 ? 3 : 2;

// Position in a ring of N stages: stage, and the parity of its current pass
// (counted up: a 64-bit modulo by 3 per use cost the issuing warp more than
// its waits).
template <int N>
struct Ring {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next() {
    if (++s == N) {
      s = 0;
      ph ^= 1;
    }
  }
};
// 32 columns of this warp's 32 TMEM lanes (the wait in the same statement).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

// One look at a barrier's phase, without waiting.
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

template <int MODE, int CG>
struct WideSmem {
  static constexpr int AST = MODE == MODE_TF32 || CG == 2 ? 4 : 3;  // A stages
  static constexpr int BST = MODE == MODE_TF32 || CG == 2 ? 4 : 3;  // B stages = A slots in tensor memory
  static constexpr uint32_t A_BYTES = BM * wide_kc<MODE>() * 8;  // boxes of 32 floats x 128 rows
  static constexpr uint32_t B_BYTES = kWideCols / CG * 128;      // hi or lo: [re 64 B | im 64 B] rows (a pair: this
                                                                 // CTA's half of the columns)
  static constexpr uint32_t BOFF = AST * A_BYTES;
  static constexpr uint32_t STAGING = 8 * 4096;                  // epilogue: two buffers of 32 rows x 64 B a warp
  static constexpr uint32_t STAGING_OFF = BOFF + BST * 2 * B_BYTES;
  static constexpr uint32_t BARS_OFF = STAGING_OFF + STAGING;
  static constexpr uint32_t BARS = 512;
  static constexpr int EC = kWideCols / 2;                // complex columns per epilogue thread
  // FP16: ring of row exponents, one entry per accumulation range. The split
  // warps run at most BST k-blocks ahead of the products and the products at
  // most one range ahead of the epilogue.
  static constexpr int XR = MODE == MODE_F16 ? 8 : 0;
  static constexpr int XRI = XR > 0 ? XR : 1;
  static constexpr uint32_t X_OFF = BARS_OFF + BARS;
  static constexpr uint32_t TOTAL = X_OFF + XR * BM + 1024;  // + alignment
  static constexpr uint32_t SLOT_COLS = 64;                  // re hi, im hi, re lo, im lo: 16 columns each
  static constexpr int NACC = kWideAcc<MODE, CG>;
  static constexpr uint32_t SLOT0 = NACC * kWideCols;        // tensor-memory columns: accumulators, then A slots
  static constexpr int SLOTS = (512 - SLOT0) / SLOT_COLS < BST ? (512 - SLOT0) / SLOT_COLS : BST;
  // one slot per B stage: the products of a k-block release both on one barrier
  static constexpr bool SLOT_IS_STAGE = SLOTS == BST;
  static_assert(SLOT0 + SLOTS * SLOT_COLS <= 512, "tensor memory");
  static_assert((2 * AST + 2 * BST + 2 * SLOTS + 2 * NACC + 2 + XR) * 8 + 16 <= BARS, "barriers and flags fit in BARS");
};

// SET: with the launch settings (TcArgs::prefetch, bit 1 of TcArgs::l2_mode). An
// instance of its own: as arguments of one kernel they cost products that leave
// them at their defaults registers and branches of the loading and storing warps
// (FP16 b256 M4096 N512 K32 1030 -> 1084 us, TF32 b64 M4096 N1024 K64 489 -> 527).
template <int MODE, int CG, bool SET>
__global__ void __launch_bounds__(kWideThreads, 1)
    tc_wide_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmBh,
                   const __grid_constant__ CUtensorMap tmBl, const __grid_constant__ CUtensorMap tmC, TcArgs a) {
  using L = WideSmem<MODE, CG>;
  constexpr int KC = wide_kc<MODE>();
  constexpr int kFoldKb = kFoldK / (2 * KC);  // k-blocks per accumulation range
  constexpr int kGroup = kWideGroup<MODE, CG>;
  static_assert(kFoldKb % kGroup == 0, "groups of k-blocks within a range");
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *afull = reinterpret_cast<uint64_t *>(smem + L::BARS_OFF);  // [AST] A stage landed
  uint64_t *aempty = afull + L::AST;   // [AST] A stage read by the split warps
  uint64_t *bfull = aempty + L::AST;   // [BST] B stage landed
  uint64_t *bempty = bfull + L::BST;       // [BST] products of the k-block retired
  uint64_t *conv = bempty + L::BST;        // [SLOTS] A split into its slot
  uint64_t *sempty_own = conv + L::SLOTS;  // [SLOTS] products that read the slot retired
  uint64_t *sempty = L::SLOT_IS_STAGE ? bempty : sempty_own;
  uint64_t *tfull = sempty_own + L::SLOTS;  // [NACC] accumulator complete for a range
  uint64_t *tempty = tfull + L::NACC;       // [NACC] drained by the epilogue
  uint64_t *drain = tempty + L::NACC;       // all products retired
  uint64_t *stall = drain + 1;         // test stall: nothing ever arrives here
  uint64_t *xfull = stall + 1;         // [XR] FP16: row exponents of a range written
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(xfull + L::XR);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  uint8_t *staging = smem + L::STAGING_OFF;
  int8_t *aexp = reinterpret_cast<int8_t *>(smem + L::X_OFF);
  auto A_raw = [&](int s) { return smem + s * L::A_BYTES; };
  auto B_hi = [&](int s) { return smem + L::BOFF + s * 2 * L::B_BYTES; };
  auto B_lo = [&](int s) { return smem + L::BOFF + s * 2 * L::B_BYTES + L::B_BYTES; };

  // (the shuffle tells the compiler that the role is uniform over the warp)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x / 32), 0), lane = threadIdx.x % 32;
  const int64_t per_batch = (int64_t)a.n_tiles_m * a.n_tiles_n;
  const int64_t n_tiles = per_batch * a.batch * a.ksplit;
  // tile walkers: CTAs, or pairs of CTAs (clusters)
  const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
  const int64_t walker = CG == 2 ? (int64_t)cluster_id_x() : (int64_t)blockIdx.x;
  const int64_t n_walkers = CG == 2 ? (int64_t)n_clusters_x() : (int64_t)gridDim.x;
  struct Tile {
    int64_t z, row0;
    int nt, rowA, rowB, ks, kb0, kb1;
  };
  auto decode = [&](int64_t t) {
    Tile d;
    d.ks = (int)(t % a.ksplit);
    t /= a.ksplit;
    d.kb0 = d.ks * a.kb_per;
    d.kb1 = min(a.kblocks, d.kb0 + a.kb_per);
    d.z = t / per_batch;
    const int64_t rem = t - d.z * per_batch;
    const int mt = (int)(rem / a.n_tiles_n);
    d.nt = (int)(rem % a.n_tiles_n);
    d.row0 = (int64_t)mt * (BM * CG) + (int64_t)rank * BM;
    d.rowA = (int)(d.z * a.M + d.row0);
    // (the last column tile may run into the next batch's rows: columns of
    // the product beyond N, which are not stored)
    d.rowB = (int)(d.z * a.NT + (int64_t)d.nt * kWideCols + (int64_t)rank * (kWideCols / CG));
    return d;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < L::AST; s++) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 4);  // one elected arrival per split warp
    }
    for (int s = 0; s < L::BST; s++) {
      mbar_init(&bfull[s], 1);
      mbar_init(&bempty[s], 1);
    }
    for (int s = 0; s < L::SLOTS; s++) {
      mbar_init(&conv[s], 4 * CG);
      mbar_init(&sempty_own[s], 1);
    }
    for (int h = 0; h < L::NACC; h++) {
      mbar_init(&tfull[h], 1);
      mbar_init(&tempty[h], 8 * CG);
    }
    mbar_init(drain, 1);
    mbar_init(stall, 1);
    for (int x = 0; x < L::XR; x++) mbar_init(&xfull[x], 4);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    // a pair allocates collectively: one warp of each CTA, the same columns
    if constexpr (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(512u));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(512u));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
  }
  tc_fence_before();
  __syncthreads();
  // a pair: the peer's barriers are initialised before anyone arrives on them
  if constexpr (CG == 2) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const unsigned long long wait_ns = g_wait_ns;
  // a wait that gives up (timeout, or an abort) also stops the peer CTA
  auto wait = [&](uint64_t *bar, uint32_t parity) {
    const bool ok = mbar_wait(bar, parity, abort_flag, wait_ns);
    if (CG == 2 && !ok) st_remote_u32(cluster_addr((const void *)abort_flag, rank ^ 1u), 1u);
    return ok;
  };
  // arrival on a barrier of the issuing CTA; commit of the products to a
  // barrier of each CTA
  auto arrive_issuer = [&](uint64_t *bar) {
    if constexpr (CG == 2)
      mbar_arrive_remote(cluster_addr(bar, 0));
    else
      mbar_arrive(bar);
  };
  auto commit = [&](uint64_t *bar) {
    if constexpr (CG == 2) {
      umma_commit_pair(cluster_addr(bar, 0));
      umma_commit_pair(cluster_addr(bar, 1));
    } else {
      umma_commit(bar);
    }
  };
  // named barriers of the MMA and waiter warps (64 threads, both whole warps)
  auto named_sync = [](int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); };
  auto named_arrive = [](int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); };
  auto named_all = [](int id, bool ok_in) {
    uint32_t all;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 q, %1, 0;\n bar.red.and.pred p, %2, 64, q;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(all)
        : "r"((uint32_t)ok_in), "r"(id)
        : "memory");
    return all != 0;
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0 && lane == 0) {
      const uint64_t stream = (a.l2_mode & 1) ? l2_evict_normal() : l2_evict_first();
      int64_t g = 0;
      Ring<L::AST> r;
      bool ok = true;
      ACursor<Tile> pc{walker, SET && a.prefetch > 0};
      auto prefetch_next = [&]() {
        if (!SET || !pc.next(n_tiles, n_walkers, decode)) return;
#pragma unroll
        for (int h = 0; h < 2 * KC / 32; h++) tma_prefetch_2d(&tmA, pc.kb * 2 * KC + 32 * h, pc.d.rowA);
      };
      for (int i = 0; SET && i < a.prefetch; i++) prefetch_next();
      for (int64_t t = walker; t < n_tiles && ok; t += n_walkers) {
        const Tile d = decode(t);
        for (int kb = d.kb0; kb < d.kb1; kb++, g++, r.next()) {
          prefetch_next();
          const int s = r.s;
          if (g >= L::AST && !wait(&aempty[s], r.ph ^ 1)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&afull[s], L::A_BYTES);
#pragma unroll
          for (int h = 0; h < 2 * KC / 32; h++)
            tma_load_2d(A_raw(s) + h * BM * 128, &tmA, kb * 2 * KC + 32 * h, d.rowA, &afull[s], stream);
        }
      }
      if (*abort_flag)
        for (int64_t q = g > L::AST ? g - L::AST : 0; q < g; q++)
          mbar_wait(&afull[q % L::AST], (uint32_t)((q / L::AST) & 1), abort_flag, kDrainNs, false);
    } else if (warp == 3 && lane == 0) {
      const uint64_t keep = l2_evict_last();
      wait_dependency();  // B is prepared
      int64_t g = 0;
      Ring<L::BST> r;
      bool ok = true;
      for (int64_t t = walker; t < n_tiles && ok; t += n_walkers) {
        const Tile d = decode(t);
        for (int kb = d.kb0; kb < d.kb1; kb++, g++, r.next()) {
          const int s = r.s;
          if (g >= L::BST && !wait(&bempty[s], r.ph ^ 1)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&bfull[s], 2 * L::B_BYTES);
          tma_load_2d(B_hi(s), &tmBh, kb * 2 * KC, d.rowB, &bfull[s], keep);
          tma_load_2d(B_lo(s), &tmBl, kb * 2 * KC, d.rowB, &bfull[s], keep);
        }
      }
      if (*abort_flag)
        for (int64_t q = g > L::BST ? g - L::BST : 0; q < g; q++)
          mbar_wait(&bfull[q % L::BST], (uint32_t)((q / L::BST) & 1), abort_flag, kDrainNs, false);
    } else if (warp == 1 && rank != 0) {
      // the pair's second CTA issues no products: it waits until the first
      // CTA's (which use its tensor and shared memory) have retired
      // (one wait for the whole launch, so its limit is long: the first CTA's
      // own waits end a launch that is stuck)
      if (lane == 0) mbar_wait(drain, 0, abort_flag, kPairNs, false);
      __syncwarp();
    } else if (warp == 1) {
      constexpr uint32_t idesc = MODE == MODE_TF32   ? idesc_tf32(kWideCols, BM * CG)
                                 : MODE == MODE_BF16 ? idesc_bf16(kWideCols, BM * CG)
                                                     : idesc_f16(kWideCols, BM * CG);
      constexpr uint32_t idesc_neg = idesc | (1u << 13);  // negate A
      // the twelve products of one half (0: D_re, 1: D_im) of the k-block in B
      // stage s and A slot sl; operand addresses advance from bases computed once
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      const uint64_t desc0 = sw128_desc(__shfl_sync(0xffffffffu, smem_u32(smem + L::BOFF), 0));
      auto issue = [&](int s, int sl, int acc_i, int h, bool first) {
        const uint32_t d_acc = tm + (uint32_t)(acc_i * kWideCols);
        const uint32_t at = tm + L::SLOT0 + (uint32_t)sl * L::SLOT_COLS;
        const uint64_t bh = desc0 + (uint64_t)(s * (2 * L::B_BYTES >> 4)), bl = bh + (L::B_BYTES >> 4);
#pragma unroll
        for (int kk = 0; kk < 2; kk++) {
#pragma unroll
          for (int im = 0; im < 2; im++) {
            // im = 0: A_re with B_re (D_re) or B_im (D_im); im = 1: A_im
            // with B_im, negated (D_re), or B_re (D_im)
            const uint32_t ah = at + (uint32_t)(im * 16 + kk * 8), al = ah + 32;
            const uint32_t bo = (uint32_t)(((im ^ h) * 64) + kk * 32) >> 4;
            const uint64_t dbh = bh + bo, dbl = bl + bo;
            const uint32_t id = (im && h == 0) ? idesc_neg : idesc;
            const uint32_t acc = !(first && kk == 0 && im == 0);
            auto mma = [&](uint32_t at_, uint64_t db, uint32_t accum) {
              if constexpr (MODE == MODE_TF32 && CG == 2)
                umma_tf32_ts_pair(d_acc, at_, db, id, accum);
              else if constexpr (MODE == MODE_TF32)
                umma_tf32_ts(d_acc, at_, db, id, accum);
              else if constexpr (CG == 2)
                umma_f16_ts_pair(d_acc, at_, db, id, accum);
              else
                umma_f16_ts(d_acc, at_, db, id, accum);
            };
            mma(ah, dbh, acc);
            mma(ah, dbl, 1);
            mma(al, dbh, 1);
          }
        }
      };
      Ring<L::BST> r;
      Ring<L::SLOTS> rs;
      Ring<L::NACC> qa[2];  // D_re's accumulator of the range, D_im's
      qa[1].next();
      uint32_t u = 0;  // units handed over
      for (int64_t t = walker; t < n_tiles; t += n_walkers) {
        const Tile d = decode(t);
        const int nkb = d.kb1 - d.kb0;
        for (int kb = 0; kb < nkb; kb += kGroup) {
          const bool first = kb % kFoldKb == 0, last = (kb + kGroup) % kFoldKb == 0 || kb + kGroup >= nkb;
          const int st0 = r.s, sl0 = rs.s;
          r.next();
          rs.next();
          const bool two = kGroup == 2 && kb + 1 < nkb;
          const int st1 = r.s, sl1 = rs.s;
          if (two) r.next(), rs.next();
#pragma unroll
          for (int h = 0; h < 2; h++) {
#pragma unroll
            for (int j = 0; j < 2; j++) {
              if (j == 1 && !two) break;
              named_sync(kBarReady + (int)(u & 1));
              tc_fence_after();
              if (elect_one()) {
                issue(j ? st1 : st0, j ? sl1 : sl0, qa[h].s, h, first && j == 0);
                if (h == 1) {
                  if (!L::SLOT_IS_STAGE) commit(&sempty[j ? sl1 : sl0]);
                  commit(&bempty[j ? st1 : st0]);
                }
                if (last && j == (two ? 1 : 0)) commit(&tfull[qa[h].s]);
              }
              __syncwarp();
              named_arrive(kBarIssued + (int)(u & 1));
              u++;
            }
          }
          if (last)
            for (int h = 0; h < 2; h++) qa[h].next(), qa[h].next();
        }
        if (!named_all(kBarTile, true)) break;
      }
      if (elect_one()) {
        commit(drain);
        mbar_wait(drain, 0, abort_flag, kDrainNs, false);
      }
      __syncwarp();
    } else if (warp == 2 && rank == 0) {
      // readiness waiter: hands the units (one k-block into one accumulator)
      // over, at most two ahead of the issuing thread, which never waits on a
      // barrier in memory itself. After a wait gives up it releases the
      // rest of the tile at once; the status reduction at the tile's end
      // stops both warps (the products issued meanwhile are discarded with
      // the call's error status).
      int64_t rg = 0;
      uint32_t u = 0;
      Ring<L::BST> r;
      Ring<L::SLOTS> rs;
      Ring<L::NACC> qa[2];
      qa[1].next();
      bool ok = true;
      if (lane == 0 && g_stall) ok = wait(stall, 0);
      for (int64_t t = walker; t < n_tiles; t += n_walkers) {
        const Tile d = decode(t);
        const int nkb = d.kb1 - d.kb0;
        for (int kb = 0; kb < nkb; kb += kGroup) {
          const bool first = kb % kFoldKb == 0, two = kGroup == 2 && kb + 1 < nkb;
#pragma unroll
          for (int h = 0; h < 2; h++) {
#pragma unroll
            for (int j = 0; j < 2; j++) {
              if (j == 1 && !two) break;
              if (lane == 0 && ok) {
                // (half-range 2 rg + h is the ring's n-th, n >= NACC)
                if (first && j == 0 && 2 * rg + h >= L::NACC) ok = wait(&tempty[qa[h].s], qa[h].ph ^ 1);
                if (h == 0 && ok) ok = (CG == 2 || wait(&bfull[r.s], r.ph)) && wait(&conv[rs.s], rs.ph);
              }
              if (h == 0) r.next(), rs.next();
              __syncwarp();
              // unit u - 2 has been issued: its ready barrier may be reused
              if (u >= 2) named_sync(kBarIssued + (int)(u & 1));
              named_arrive(kBarReady + (int)(u & 1));
              u++;
            }
          }
          if ((kb + kGroup) % kFoldKb == 0 || kb + kGroup >= nkb) {
            rg++;
            for (int h = 0; h < 2; h++) qa[h].next(), qa[h].next();
          }
        }
        ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
        if (!named_all(kBarTile, ok)) break;
      }
      // take the last "issued" arrivals, so that every barrier generation
      // completes before the CTA exits
      for (uint32_t q = u > 2 ? u - 2 : 0; q < u; q++) named_sync(kBarIssued + (int)(q & 1));
    }
  } else if (warp < 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 120;");
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + L::SLOT0;
    int64_t g = 0, rg = 0;
    Ring<L::AST> ra;
    Ring<L::BST> rb;
    Ring<L::SLOTS> rs;
    int range_se = 0;
    bool ok = true;
    // a row of a stage: 16-byte chunk c (two complex values) sits at chunk
    // c ^ (row & 7) of its box
    constexpr int NCH = KC / 2;  // chunks of a row: 8 (TF32) or 16 in two boxes
    uint4 v[NCH];
    auto chunk = [&](int st, int c) {
      return reinterpret_cast<const uint4 *>(A_raw(st) + (c >> 3) * BM * 128 + row * 128)[(c & 7) ^ (row & 7)];
    };
    auto fetch = [&](int st) {
#pragma unroll
      for (int c = 0; c < NCH; c++) v[c] = chunk(st, c);
    };
    for (int64_t tile = walker; tile < n_tiles && ok; tile += n_walkers) {
      const Tile d = decode(tile);
      const int nkb = d.kb1 - d.kb0;
      bool loaded = false;  // v holds the k-block already
      for (int kb = 0; kb < nkb; kb++, g++, ra.next(), rb.next(), rs.next()) {
        const int as = ra.s, s = rb.s;
        const uint32_t ts = tq + (uint32_t)rs.s * L::SLOT_COLS;
        if (!loaded && !(ok = wait(&afull[as], ra.ph))) break;
        if (!loaded) fetch(as);
        if (MODE == MODE_F16 && kb % kFoldKb == 0) {
          // the largest magnitude of the row's values of the whole range (its
          // other k-blocks' stages are waited for here) sets the exponent
          float m = 0.f;
          auto mag = [&](const uint4 &w) {
            m = fmaxf(fmaxf(m, fmaxf(fabsf(__uint_as_float(w.x)), fabsf(__uint_as_float(w.y)))),
                      fmaxf(fabsf(__uint_as_float(w.z)), fabsf(__uint_as_float(w.w))));
          };
#pragma unroll
          for (int c = 0; c < NCH; c++) mag(v[c]);
          Ring<L::AST> rj = ra;
          for (int j = 1; j < kFoldKb && kb + j < nkb; j++) {
            rj.next();
            if (!wait(&afull[rj.s], rj.ph)) {
              ok = false;
              break;
            }
#pragma unroll
            for (int c = 0; c < NCH; c++) mag(chunk(rj.s, c));
          }
          if (!ok) break;
          range_se = f16_scale_exp(__float_as_uint(m));
          aexp[(int)(rg % L::XRI) * BM + row] = (int8_t)range_se;
        }
        // the slot is free once the products that read it have retired
        if (g >= L::SLOTS && !wait(&sempty[rs.s], rs.ph ^ 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (MODE == MODE_TF32) {
          uint32_t hr[16], hi[16];
#pragma unroll
          for (int c = 0; c < 8; c++) {
            hr[2 * c] = split_hi(v[c].x);
            hi[2 * c] = split_hi(v[c].y);
            hr[2 * c + 1] = split_hi(v[c].z);
            hi[2 * c + 1] = split_hi(v[c].w);
          }
          tmem_st16(ts, hr);
          tmem_st16(ts + 16, hi);
#pragma unroll
          for (int c = 0; c < 8; c++) {
            hr[2 * c] = __float_as_uint(__uint_as_float(v[c].x) - __uint_as_float(hr[2 * c]));
            hi[2 * c] = __float_as_uint(__uint_as_float(v[c].y) - __uint_as_float(hi[2 * c]));
            hr[2 * c + 1] = __float_as_uint(__uint_as_float(v[c].z) - __uint_as_float(hr[2 * c + 1]));
            hi[2 * c + 1] = __float_as_uint(__uint_as_float(v[c].w) - __uint_as_float(hi[2 * c + 1]));
          }
          tmem_st16(ts + 32, hr);
          tmem_st16(ts + 48, hi);
        } else {
          const float sa = MODE == MODE_F16 ? pow2i(range_se) : 1.f;
#pragma unroll
          for (int h = 0; h < 2; h++) {
            uint32_t hr[8], hi[8], lr[8], li[8];
#pragma unroll
            for (int c = 0; c < 8; c++) {
              const uint4 w = v[8 * h + c < NCH ? 8 * h + c : 0];
              const float x0 = __uint_as_float(w.x), y0 = __uint_as_float(w.y), x1 = __uint_as_float(w.z),
                          y1 = __uint_as_float(w.w);
              if (MODE == MODE_F16) {
                split_f16x2(x0 * sa, x1 * sa, hr[c], lr[c]);
                split_f16x2(y0 * sa, y1 * sa, hi[c], li[c]);
              } else {
                split_bf16x2(x0, x1, hr[c], lr[c]);
                split_bf16x2(y0, y1, hi[c], li[c]);
              }
            }
            tmem_st8(ts + (uint32_t)(8 * h), hr);
            tmem_st8(ts + (uint32_t)(16 + 8 * h), hi);
            tmem_st8(ts + (uint32_t)(32 + 8 * h), lr);
            tmem_st8(ts + (uint32_t)(48 + 8 * h), li);
          }
        }
        // the row has been split: the stage can be loaded again (the fence
        // orders the reads before the copy that overwrites them; without it
        // reads still in flight saw the next rows)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&aempty[as]);
        // the next row is fetched while the stores to tensor memory complete,
        // if it has landed
        Ring<L::AST> rn = ra;
        rn.next();
        loaded = kb + 1 < nkb && __all_sync(0xffffffffu, mbar_test_wait(&afull[rn.s], rn.ph));
        if (loaded) fetch(rn.s);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        const bool last = kb % kFoldKb == kFoldKb - 1 || kb == nkb - 1;
        if (lane == 0) {
          // a pair: the arrival also says that this CTA's half of B has landed
          if (CG == 2 && !wait(&bfull[s], rb.ph)) ok = false;
          if (ok) arrive_issuer(&conv[rs.s]);
          if (MODE == MODE_F16 && last) mbar_arrive(&xfull[rg % L::XRI]);
        }
        if (CG == 2 && !__shfl_sync(0xffffffffu, (int)ok, 0)) {
          ok = false;
          break;
        }
        if (last) rg++;
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    // epilogue: warps 8..11 take complex columns 0..63 of the tile, 12..15
    // the rest; each thread sums its part of a row over the ranges
    constexpr int EC = L::EC;
    const int e = warp - 8;
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const int c0 = (e >> 2) * EC;
    const bool streaming = !SET || (a.l2_mode & 2) != 0;  // C evict first
    uint8_t *buf0 = staging + e * 4096;
    wait_dependency();  // the column scales are written
    Ring<L::NACC> qe;
    int64_t rg = 0;
    bool ok = true;
    for (int64_t tile = walker; tile < n_tiles && ok; tile += n_walkers) {
      const Tile d = decode(tile);
      const int64_t n0 = (int64_t)d.nt * kWideCols + c0;  // first complex column of this warp
      // per-column values (scatter offsets, FP16 scales): columns lane and
      // lane + 32 in this lane's registers, read by shuffles
      float scl[2] = {0.f, 0.f};
      if (MODE == MODE_F16) {
#pragma unroll
        for (int u = 0; u < 2; u++)
          if (n0 + lane + 32 * u < a.N) scl[u] = a.cscale[d.z * a.N + n0 + lane + 32 * u];
      }
      float re[EC], im[EC];
#pragma unroll
      for (int j = 0; j < EC; j++) re[j] = im[j] = 0.f;
      const int nkb = d.kb1 - d.kb0;
      for (int r0 = 0; r0 < nkb; r0 += kFoldKb, rg++) {
        float ua = 1.f;
#pragma unroll
        for (int h = 0; h < 2; h++) {
          if (!ok) break;
          if (!wait(&tfull[qe.s], qe.ph)) {
            ok = false;
            break;
          }
          if (MODE == MODE_F16 && h == 0) {
            // (released before the range's products were issued)
            if (!wait(&xfull[rg % L::XRI], (uint32_t)((rg / L::XRI) & 1))) {
              ok = false;
              break;
            }
            ua = pow2i(-(int)aexp[(int)(rg % L::XRI) * BM + row]);
          }
          tc_fence_after();
          const uint32_t taddr = tmem + (uint32_t)(qe.s * kWideCols + c0) + ((uint32_t)(q * 32) << 16);
#pragma unroll
          for (int c = 0; c < EC; c += 32) {
            uint32_t r[32];
            tmem_ld32(taddr + (uint32_t)c, r);
#pragma unroll
            for (int j = 0; j < 32; j++) {
              float &x = h ? im[c + j] : re[c + j];
              if (MODE == MODE_F16)
                x = fmaf(__uint_as_float(r[j]), ua, x);
              else
                x += __uint_as_float(r[j]);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) arrive_issuer(&tempty[qe.s]);
          qe.next();
        }
        if (!ok) break;
      }
      if (!ok) break;
      // FP16: columns c .. c + 7 times their scales, chunk by chunk as they
      // are stored (all 64 at once need more registers than there are)
      auto scale8 = [&](int c) {
        if (MODE == MODE_F16) {
          asm volatile("" ::: "memory");
#pragma unroll
          for (int j = c; j < c + 8; j++) {
            const float u = __shfl_sync(0xffffffffu, scl[j >> 5], j & 31);
            re[j] *= u;
            im[j] *= u;
          }
        }
      };
      if (a.scatter) {
        int64_t off[2] = {0, 0};  // offsets of columns lane and lane + 32
        const bool linear = a.scatter == 3;  // row-major partials of a split K
#pragma unroll
        for (int u = 0; u < 2; u++)
          off[u] = linear ? n0 + lane + 32 * u : scatter_bits(n0 + lane + 32 * u, a.sc.nn, a.sc.pn);
        const int64_t om = linear ? d.ks * a.split_stride + d.z * a.sC + (d.row0 + row) * a.N
                                  : scatter_bits(d.z, a.sc.nb, a.sc.pb) +
                                        scatter_bits(d.row0 + row, a.sc.nm, a.sc.pm);
        if (a.scatter >= 2) {
          // as in tc_split3_kernel: 32 rows x 8 complex through a swizzled
          // buffer, then 8 rows x 4 column pairs (16 bytes) per store
          int64_t om_u[4];
#pragma unroll
          for (int u = 0; u < 4; u++) om_u[u] = __shfl_sync(0xffffffffu, om, 8 * u + (lane >> 2));
#pragma unroll
          for (int c = 0; c < EC; c += 8) {
            scale8(c);
            if (n0 + c < a.N) {  // N is a multiple of 8 here
              // (alternating buffers: the rows of two chunks ago were read
              // before the barrier of the chunk between)
              uint8_t *buf = buf0 + (c & 8) * 256;
#pragma unroll
              for (int j = 0; j < 4; j++)
                *reinterpret_cast<float4 *>(buf + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) =
                    make_float4(re[c + 2 * j], im[c + 2 * j], re[c + 2 * j + 1], im[c + 2 * j + 1]);
              __syncwarp();
              const int64_t col = __shfl_sync(0xffffffffu, off[c >> 5], (c & 31) + 2 * (lane & 3));
#pragma unroll
              for (int u = 0; u < 4; u++) {
                const int rr = 8 * u + (lane >> 2);
                const uint4 w =
                    *reinterpret_cast<const uint4 *>(buf + rr * 64 + (((lane & 3) ^ ((rr >> 1) & 3)) << 4));
                store_c(reinterpret_cast<uint4 *>(a.C + om_u[u] + col), w, streaming);
              }
            }
          }
          __syncwarp();
        } else {
#pragma unroll
          for (int j = 0; j < EC; j++) {
            if (j % 8 == 0) scale8(j);
            const int64_t col = __shfl_sync(0xffffffffu, off[j >> 5], j & 31);
            if (n0 + j < a.N) store_c(a.C + om + col, make_float2(re[j], im[j]), streaming);
          }
        }
      } else if (a.tma_store) {
        const int y = (int)(d.z * a.M + d.row0 + q * 32);
        // chunks use the two buffers in turn and a tile starts over at the
        // first; a warp's last chunk of a tile used the first as well only with
        // an odd number of chunks in a row of C (waiting there in every tile
        // costs what the stores of short K overlap: FP16 b256 M4096 N512 K32
        // 1024 -> 1081 us, so 1030)
        const bool odd = ((a.N + 7) >> 3) & 1;
#pragma unroll
        for (int c = 0; c < EC; c += 8) {
          scale8(c);
          if (n0 + c < a.N) {
            uint8_t *buf = buf0 + (c & 8) * 256;
            // the store before the last has read this buffer (the first chunk of
            // a tile: every store has, where the last store of the tile before
            // may have used this buffer too)
            if (lane == 0) {
              if (c == 0 && odd)
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
              else
                asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 4; j++)
              *reinterpret_cast<float4 *>(buf + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) =
                  make_float4(re[c + 2 * j], im[c + 2 * j], re[c + 2 * j + 1], im[c + 2 * j + 1]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
              asm volatile(
                  "cp.async.bulk.tensor.2d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%1, %2}], [%3], %4;" ::"l"(
                      (uint64_t)&tmC),
                  "r"((int)(2 * (n0 + c))), "r"(y), "r"(smem_u32(buf)), "l"(streaming ? l2_evict_first() : l2_evict_normal())
                  : "memory");
              asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
          }
        }
      } else {
        float2 *crow = a.C + d.ks * a.split_stride + d.z * a.sC + (d.row0 + row) * a.N;
#pragma unroll
        for (int j = 0; j < EC; j++) {
          if (j % 8 == 0) scale8(j);
          if (n0 + j < a.N) store_c(crow + n0 + j, make_float2(re[j], im[j]), streaming);
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && a.err) atomicExch(a.err, 1);
  // a pair: neither CTA leaves (or frees tensor memory) while the other may
  // still arrive on its barriers
  if constexpr (CG == 2) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (CG == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

// B (columns of K complex values) -> planes, hi and lo: a column's row holds,
// per k-block of wide_kc values, the real parts (64 bytes), then the
// imaginary parts; the last k-block is padded with zeros. One group of G
// threads (a warp or the block) per column. FP16: the column is scaled by its
// own power of two (largest magnitude to [2^14, 2^15), so one pass of the
// block over B finds the exponent and splits), and cscale receives the
// inverse, applied per column in the product's epilogue.
template <int MODE, int G>
__global__ void __launch_bounds__(256)
    prep_planes_kernel(const float2 *__restrict__ B, void *__restrict__ Bh_, void *__restrict__ Bl_,
                       float *__restrict__ cscale, int64_t cols, int64_t K, int64_t Kp, int vec, int *clear) {
  launch_dependents();
  if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0;
  static_assert(G == 32 || G == 256, "a warp or the block per column");
  constexpr int V = MODE == MODE_TF32 ? 2 : 4;  // complex values a thread takes at a time
  constexpr int KC = wide_kc<MODE>();
  __shared__ uint32_t wm[8];
  const int t = threadIdx.x % G;
  const int64_t groups = (int64_t)gridDim.x * (256 / G);
  for (int64_t col = blockIdx.x * (int64_t)(256 / G) + threadIdx.x / G; col < cols; col += groups) {
    const float2 *b = B + col * K;
    auto load = [&](int64_t k, float2 (&x)[V]) {
      if (vec) {
#pragma unroll
        for (int j = 0; j < V; j += 2) {
          const float4 w = *reinterpret_cast<const float4 *>(b + k + j);
          x[j] = make_float2(w.x, w.y);
          x[j + 1] = make_float2(w.z, w.w);
        }
      } else {
#pragma unroll
        for (int j = 0; j < V; j++) x[j] = b[k + j];
      }
    };
    float sb = 1.f;
    if (MODE == MODE_F16) {
      uint32_t m = 0;
      for (int64_t k = V * t; k < K; k += V * G) {
        float2 x[V];
        load(k, x);
#pragma unroll
        for (int j = 0; j < V; j++)
          m = max(m, max(__float_as_uint(x[j].x) & 0x7fffffffu, __float_as_uint(x[j].y) & 0x7fffffffu));
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (G == 256) {
        __syncthreads();  // the previous column's maxima have been read
        if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; w++) m = max(m, wm[w]);
      }
      const int s = f16_scale_exp(m);
      sb = pow2i(s);
      if (t == 0) cscale[col] = pow2i(-s);
    }
    for (int64_t k = V * t; k < Kp; k += V * G) {
      float2 x[V];
      if (k < K) {
        load(k, x);
      } else {
#pragma unroll
        for (int j = 0; j < V; j++) x[j] = make_float2(0.f, 0.f);
      }
      const int64_t o = col * 2 * Kp + (k / KC) * 2 * KC + k % KC;  // real parts; imaginary parts at + KC
      if (MODE == MODE_TF32) {
        uint32_t *Bh = static_cast<uint32_t *>(Bh_), *Bl = static_cast<uint32_t *>(Bl_);
        const uint32_t r0 = __float_as_uint(x[0].x), r1 = __float_as_uint(x[1].x), i0 = __float_as_uint(x[0].y),
                       i1 = __float_as_uint(x[1].y);
        *reinterpret_cast<uint2 *>(Bh + o) = make_uint2(split_hi(r0), split_hi(r1));
        *reinterpret_cast<uint2 *>(Bh + o + KC) = make_uint2(split_hi(i0), split_hi(i1));
        *reinterpret_cast<uint2 *>(Bl + o) = make_uint2(split_lo(r0), split_lo(r1));
        *reinterpret_cast<uint2 *>(Bl + o + KC) = make_uint2(split_lo(i0), split_lo(i1));
      } else {
        uint16_t *Bh = static_cast<uint16_t *>(Bh_), *Bl = static_cast<uint16_t *>(Bl_);
        uint32_t hr[2], lr[2], hi[2], li[2];
#pragma unroll
        for (int j = 0; j < 2; j++) {
          const float2 p = x[(2 * j) % V], s = x[(2 * j + 1) % V];
          if (MODE == MODE_F16) {
            split_f16x2(p.x * sb, s.x * sb, hr[j], lr[j]);
            split_f16x2(p.y * sb, s.y * sb, hi[j], li[j]);
          } else {
            split_bf16x2(p.x, s.x, hr[j], lr[j]);
            split_bf16x2(p.y, s.y, hi[j], li[j]);
          }
        }
        *reinterpret_cast<uint2 *>(Bh + o) = make_uint2(hr[0], hr[1]);
        *reinterpret_cast<uint2 *>(Bh + o + KC) = make_uint2(hi[0], hi[1]);
        *reinterpret_cast<uint2 *>(Bl + o) = make_uint2(lr[0], lr[1]);
        *reinterpret_cast<uint2 *>(Bl + o + KC) = make_uint2(li[0], li[1]);
      }
    }
  }
}
