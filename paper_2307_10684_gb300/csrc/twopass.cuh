// Mode products of an operator's first two directions in one launch of two
// dependent passes (part of tc.cu, inside its anonymous namespace).
//
// tc_fused_kernel keeps the intermediate in TMEM, but computes it again for
// every 128-row tile of x2 whose support reaches it: with supports as wide as
// the grid that is n2 / 128 times.  Here the x1 product is written once, as
// BF16 pieces, and read by the x2 tiles of the same launch; nothing is
// computed twice, and the work spreads over any number of SMs.
//
// Passes.  Every product reads its data operand as rows [M][K = n_mu]
// (flattened over the slabs of the other directions, so that only the last
// tile is padded) and Phi as the N operand, N tile = any multiple of 16 up to
// 256.  The x1 product writes [slab][j1][i2], the x2 product the natural
// [slab][j2][j1]; both are transposed within a slab, so TMEM lanes (rows) are
// contiguous in memory.  The x2 tiles wait, per tile, for the x1 tiles they
// read (counters in global memory).  In 3D the x3 product follows as a launch
// of its own on the natural-layout pieces, read MN-major.
//
// Precision: the same three BF16 pieces, six products and one FP32 accumulator
// per output as in every other kernel here.
//
// Tile width.  An MMA takes 99 clocks here whatever its N up to 128, and about
// N / 2 beyond (measured: 48 ns apart at N = 32, 80 and 128).  So of tiles that
// contract over the same range the widest is the cheapest per output: 136^3
// runs at 145 us a step with one tile of 144 columns, 163 with two of 80
// (192^3 296 / 312; 160^3 190 / 185, where a tile's latencies bound: the
// tensor pipe is busy 28% of the launch, no memory above 36%).  Beyond 256
// columns 128-wide tiles with ranges of their own win, and narrower tiles
// serve to spread small grids over more SMs (tp_geo).

constexpr int kTpBK = 32;                          // K values per stage (64-byte rows)
constexpr int kTpPieceA = kBM * 64;                // one piece of X's tile
constexpr int kTpTileA = kPieces * kTpPieceA;
// WIDE: tiles of more than 128 columns; one piece of Phi's tile has room for
// 256 rows, else 128 (the distance between pieces is a constant either way)
template <bool WIDE>
struct TpCfg {
  static constexpr int BN = WIDE ? 256 : 128;
  static constexpr int PIECE_B = BN * 64;
  static constexpr int STAGE = kTpTileA + kPieces * PIECE_B;  // 72 or 48 KB
  static constexpr int STAGES = WIDE ? 3 : 4;
  static constexpr int SMEM = STAGES * STAGE + 1024;
};
constexpr int kTpSched = 4;                        // units announced ahead
constexpr int kTpMaxSeq = 16;

// One product of one solve.
struct alignas(128) TpPass {
  CUtensorMap amap[2];       // X pieces [3][M][K]; the x3 product: [3][K][M]
  // Phi pieces [3][N][K]: boxes of bn rows of one piece per component, then
  // of 128 (bn > 128: 256) rows of all three (full tiles: one copy, not three)
  CUtensorMap bmap[4];
  // K blocks [first, end) of each group of kg 128-row groups of Phi, per
  // component: the union of their column supports (the group, not the tile,
  // decides, so that every tile width accumulates an output over the same
  // values in the same order)
  uint8_t kb[2][32][2];
  __nv_bfloat16* outp[2];    // pieces out [3][N M] (null: FP32 update)
  float* outf[2];
  const float* base[2];
  float* lo[2];              // compensated state: low-order words
  double* ind;               // indicators (last product of a step)
  const int64_t* ind_ctr;
  int ind_k, ind_n1, ind_n2;
  float alpha;
  int M, N, K, R;            // rows, columns, contraction, rows per slab
  int tiles_m, tn, bn;       // row tiles, column tiles, columns per tile (multiple of 16)
  int kg_log2;               // log2 of the 128-row groups of Phi whose supports a tile takes together
  uint32_t per_mul;          // 2^32 / (2 tn) + 1
  // counters [2][slabs][dep_tn] of finished x1 tiles: in 2D one per x1 column
  // tile (j1), in 3D one per slab; dep_r: the x1 pass's rows per slab,
  // dep_want: tiles per counter and overlapping row tile
  uint32_t* dep;
  int dep_tn, dep_r, dep_want, slabs;
};
struct TpOp {
  TpPass p[2];
};
struct TpLaunch {
  TpOp one;                  // one solve
  const TpOp* desc;          // or [nsolves] in device memory
  const int* ustart;         // [npass][nsolves + 1]
  int nsolves, npass;
  int nunits;                // all passes
  // order of the units: segment k holds tickets [seq_end[k-1], seq_end[k]) and
  // covers units seq_first[k].. of pass seq_pass[k]
  int nseq;
  int seq_end[kTpMaxSeq], seq_first[kTpMaxSeq], seq_pass[kTpMaxSeq];
  uint32_t* ctl;             // two-pass launches: ticket, CTAs done, then the dep counters
  int nctl;                  // words to clear at the end
  int ahead;                 // units a CTA may hold claimed beyond the one it loads
  int clear;                 // 1: no row kernels between the launches: claim only after the
                             // previous kernel has completed, and clear ctl at the end
  int* err;
};

// A unit, decoded once by the claiming thread and announced through shared
// memory (decoding takes a lone thread about 0.7 us, a third of a tile's MMAs).
struct TpUnit {
  const TpPass* d;           // null: no more units
  int c, mt, nt, pass, kb0, kb1, bn;
};
// x / d by the multiplier m = 2^32 / d + 1 (exact for x d < 2^32, else off by one up)
__device__ __forceinline__ int tp_div(int x, int d, uint32_t m) {
  const int q = (int)__umulhi((uint32_t)x, m);
  return q * d > x ? q - 1 : q;
}
__device__ __forceinline__ TpUnit tp_decode(const TpLaunch& L, int pass, int r) {
  TpUnit w;
  w.pass = pass;
  if (L.desc == nullptr) {
    w.d = &L.one.p[pass];
  } else {
    const int* us = L.ustart + pass * (L.nsolves + 1);
    const int s = find_segment(us, L.nsolves, r);
    w.d = &L.desc[s].p[pass];
    r -= __ldg(us + s);
  }
  const int per = 2 * w.d->tn;
  w.mt = tp_div(r, per, w.d->per_mul);
  r -= w.mt * per;
  w.c = r >= w.d->tn ? 1 : 0;
  w.nt = r - w.c * w.d->tn;
  w.bn = w.d->bn;
  const int g = ((w.nt * w.bn) >> 7) >> w.d->kg_log2;
  w.kb0 = w.d->kb[w.c][g][0];
  w.kb1 = w.d->kb[w.c][g][1];
  return w;
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async;" ::: "memory");
}
// Row tiles of the x1 pass (rows per slab r) that overlap slab s.
__device__ __forceinline__ int tp_slab_tiles(int s, int r) {
  return ((s + 1) * r - 1) / kBM - s * r / kBM + 1;
}
// Waits (bounded) until the x1 tiles that an x2 tile reads are complete.
// seen: the last counter found complete by this thread (its address: in a batch
// every solve has counters of its own, so an index would not tell two apart).
__device__ __forceinline__ bool tp_wait_dep(const TpUnit& w, const uint32_t*& seen) {
  const TpPass* d = w.d;
  const int m0 = w.mt * kBM, m1 = min(m0 + kBM, d->M) - 1;
  int s0 = 0, s1 = 0, t0 = 0, t1 = 0;
  if (d->slabs > 1) {
    s0 = m0 / d->R;
    s1 = m1 / d->R;
  } else {
    const int bn1 = w.d[-1].bn;        // the x1 pass's descriptor precedes the x2 pass's
    t0 = m0 / bn1;
    t1 = m1 / bn1;
  }
  const uint64_t start = globaltimer();
  bool fresh = false;
  for (int s = s0; s <= s1; ++s) {
    const uint32_t want = (uint32_t)(d->dep_want * tp_slab_tiles(s, d->dep_r));
    const uint32_t* row = d->dep + (w.c * d->slabs + s) * d->dep_tn;
    for (int t = t0; t <= t1; ++t) {
      if (row + t == seen) continue;
      while (ld_acquire(row + t) < want)
        if (globaltimer() - start > kWaitNs) return false;
      seen = row + t;
      fresh = true;
    }
  }
  if (fresh) fence_proxy_async();  // the pieces were written by ordinary stores of this launch
  return true;
}

// 8 columns of an accumulator (valid after tmem_wait_ld() and tp_fence()).
__device__ __forceinline__ void tp_ld(uint32_t ta, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(ta));
}
// Orders every later use of r after the preceding tmem_wait_ld().
__device__ __forceinline__ void tp_fence(uint32_t (&r)[8]) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                 "+r"(r[7])
               :
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Persistent kernel, one CTA per SM.  Warp 3 claims units, waits for what
// they read and announces them, up to four ahead (claiming, decoding and the
// counter's round trip take a lone thread 1 to 3 us a unit; in the loading
// thread they left the ring empty at every unit), warp 0 loads by TMA, warp 1
// issues the MMAs (accumulators of two units in TMEM, up to 256 columns
// each), warp 2 publishes finished x1 tiles, warps 4-19 run the
// epilogue: eight warps for the even and eight for
// the odd units, each a lane quarter and every other 16 columns.  (An
// epilogue is a chain of latencies, the unit's scales, its base, its
// accumulator, its stores, of about 2.5 us against 2 us of MMAs on a 128-wide
// tile with K = 256; with two groups two of them overlap.  The publishing
// thread waits for the tile's stores to be acknowledged, about 1 us, which
// would otherwise stop an epilogue warp.)
//
// Units of a two-pass launch are claimed from a counter, in an order in
// which a unit reads only what earlier units write: whatever subset of the
// grid is resident, the lowest incomplete unit is always running and never
// waits, so the waits end without any assumption on co-residency (two plans
// may step on two streams).  A step's two operators have a set of counters
// each (L.ctl); the row kernel that writes one's input clears the other's, a
// whole kernel before that is claimed from (pw_open); a launch that follows
// another of its kind directly (L.clear) has its last CTA clear its own.
//
// EPI: 0 = plain update or pieces, 1 = compensated state, 2 = the step's
// indicators too (separate instantiations: the extra live state would cost
// the plain epilogue registers).
constexpr int kTpEpi = 8;     // epilogue warps of a unit; two such groups
constexpr int kTpThreads = 128 + 2 * 32 * kTpEpi;
// AMN: X is read MN-major (the x3 product).  WIDE: see TpCfg.
// (EPI 0 is bounded to 64 registers, as for 1024 threads, so that a block of the row kernels
// before and after fits beside this kernel's CTA and the launches overlap.)
template <int EPI, bool AMN, bool WIDE>
__global__ void __launch_bounds__(EPI == 0 ? 1024 : kTpThreads, 1) tp_kernel(const __grid_constant__ TpLaunch L) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t full[8], empty[8], acc_full[2], acc_empty[2], stored[2];
  __shared__ uint64_t sched_full[kTpSched], sched_empty[kTpSched], drain;
  __shared__ TpUnit sched_unit[kTpSched];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag, units_issued;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  using Cfg = TpCfg<WIDE>;
  constexpr int stages = Cfg::STAGES;
  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kTpEpi + (L.npass > 1 ? 1 : 0));
      mbar_init(&stored[b], kTpEpi);
    }
    for (int b = 0; b < kTpSched; ++b) {
      mbar_init(&sched_full[b], 1);
      mbar_init(&sched_empty[b], 3 + kTpEpi);
    }
    mbar_init(&drain, 1);
    abort_flag = 0;
    units_issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* abort_v = &abort_flag;
  const bool dynamic = L.npass > 1;
  auto fail = [&](int code) {
    atomicCAS(L.err, 0, code);
    *abort_v = 1;
  };
  // the announced unit k (d null: no more units, or an abort); for one thread
  auto next_unit = [&](uint32_t k) -> TpUnit {
    const int sl = k % kTpSched;
    TpUnit w;
    w.d = nullptr;
    if (!mbar_wait(&sched_full[sl], (k / kTpSched) & 1)) {
      fail(kErrTimeoutFull);
      return w;
    }
    w = sched_unit[sl];
    mbar_arrive(&sched_empty[sl]);
    return w;
  };

  if (warp == 3 && lane == 0) {
    // ---------------- units.  The counters were cleared by a kernel that was
    // complete before the previous one let this one in, and only this launch
    // adds to them, so neither the claims nor the waits for x1 tiles wait for
    // the previous kernel
    if (dynamic && L.clear) pdl_wait();
    const uint32_t* seen = nullptr;
    uint32_t t = blockIdx.x;
    for (uint32_t k = 0;; ++k, t += gridDim.x) {
      TpUnit w;
      w.d = nullptr;
      // a unit is claimed when the loads of the one L.ahead before the last
      // are issued: claims too far ahead would leave CTAs that start late
      // (behind the previous kernel's last blocks) without work
      if (dynamic) {
        const uint64_t t0 = globaltimer();
        while (*(volatile int*)&units_issued < (int)k - L.ahead && !*abort_v)
          if (globaltimer() - t0 > kWaitNs) fail(kErrTimeoutEmpty);
        t = atomicAdd(L.ctl, 1u);
      }
      if (t < (uint32_t)L.nunits && !*abort_v) {
        int q = 0;
        while (t >= (uint32_t)L.seq_end[q]) ++q;
        w = tp_decode(L, L.seq_pass[q], L.seq_first[q] + (int)t - (q ? L.seq_end[q - 1] : 0));
        if (w.pass == 1 && !tp_wait_dep(w, seen)) {
          fail(kErrTimeoutDone);
          w.d = nullptr;
        }
      }
      // announce; after the last unit both epilogue groups get an end mark
      bool lost = false;
      for (uint32_t e = k; e <= (w.d ? k : k + 1) && !lost; ++e) {
        const int sl = e % kTpSched;
        lost = e >= kTpSched && !mbar_wait(&sched_empty[sl], (e / kTpSched - 1) & 1);
        if (lost) break;
        sched_unit[sl] = w;
        mbar_arrive(&sched_full[sl]);
      }
      if (lost) fail(kErrTimeoutEmpty);  // the readers gave up: nothing is announced any more
      if (lost || !w.d) break;
    }
  } else if (warp == 0 && lane == 0) {
    // ---------------- loads.  Ring position: slot, times the ring has been
    // passed (no divisions in the issue loops: one costs a lone thread as
    // much as two MMAs)
    int ps = 0;
    uint32_t pround = 0;
    bool waited = false, stop = false;
    for (uint32_t k = 0; !stop; ++k) {
      const TpUnit w = next_unit(k);
      if (!w.d) break;
      const CUtensorMap* ma = &w.d->amap[w.c];
      const CUtensorMap* mb = &w.d->bmap[w.c];
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)ma) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)mb) : "memory");
      const uint32_t bytes = (uint32_t)(kTpTileA + w.bn * kPieces * 64);
      const int m0 = w.mt * kBM, n0 = w.nt * w.bn;
      auto load_phi = [&](int s, int kb) {  // the pieces at fixed distances, whatever the tile width
        uint8_t* st = smem + s * Cfg::STAGE + kTpTileA;
        mbar_arrive_expect_tx(&full[s], bytes);
        if (w.bn == Cfg::BN) {
          tma_load_3d(st, &w.d->bmap[2 + w.c], &full[s], kb * kTpBK, n0, 0);
        } else {
          tma_load_3d(st, mb, &full[s], kb * kTpBK, n0, 0);
          tma_load_3d(st + Cfg::PIECE_B, mb, &full[s], kb * kTpBK, n0, 1);
          tma_load_3d(st + 2 * Cfg::PIECE_B, mb, &full[s], kb * kTpBK, n0, 2);
        }
      };
      int kpre = w.kb0;
      if (!waited) {  // Phi is plan data: its first stages need not wait for the previous kernel
        for (; kpre < min(w.kb1, w.kb0 + stages); ++kpre) load_phi(kpre - w.kb0, kpre);
        pdl_wait();
        waited = true;
      }
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        const int s = ps;
        if (*abort_v || (pround > 0 && !mbar_wait(&empty[s], (pround - 1) & 1))) {
          fail(kErrTimeoutEmpty);
          stop = true;
          break;
        }
        if (++ps == stages) {
          ps = 0;
          ++pround;
        }
        uint8_t* st = smem + s * Cfg::STAGE;
        if (kb >= kpre) load_phi(s, kb);
        if (AMN) {
          tma_load_3d(st, ma, &full[s], m0, kb * kTpBK, 0);
          tma_load_3d(st + kTpTileA / 2, ma, &full[s], m0 + 64, kb * kTpBK, 0);
        } else {
          tma_load_3d(st, ma, &full[s], kb * kTpBK, m0, 0);
        }
      }
      *(volatile int*)&units_issued = (int)k + 1;
    }
    if (!waited) pdl_wait();
    // the last loads must have landed before exit (on an abort a stage may
    // lack its X part: the wait then runs out, by when the copies have long
    // landed)
    for (int s = 0; s < stages; ++s) {
      const uint32_t uses = pround + (s < ps ? 1u : 0u);  // loads into slot s
      if (uses > 0) mbar_wait(&full[s], (uses - 1) & 1);
    }
    if (stop) mbar_wait(&full[ps], pround & 1);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer.  Every distance inside a stage is a
    // constant, so that a descriptor is the stage's plus an immediate (with
    // run-time distances an MMA took 99 clocks to issue, whatever its width)
    int ms = 0;  // ring slot and parity
    uint32_t mpar = 0;
    bool stop = false;
    const uint64_t dA0 = AMN ? mnmajor_desc128(smem_u32(smem), kTpTileA / 2, 1024) : kmajor_desc<64>(smem_u32(smem));
    const uint64_t dB0 = kmajor_desc<64>(smem_u32(smem) + kTpTileA);
    for (uint32_t k = 0; !stop; ++k) {
      const TpUnit w = next_unit(k);
      if (!w.d) break;
      const int slot = k & 1;
      if (k >= 2 && !mbar_wait(&acc_empty[slot], (k / 2 - 1) & 1)) {
        fail(kErrTimeoutDone);
        break;
      }
      tc_fence_after();
      const uint32_t idesc = idesc_bf16(kBM, w.bn) | (AMN ? 1u << 15 : 0u);
      const uint32_t dt = tmem + (uint32_t)(slot * 256);
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        const int s = ms;
        if (!mbar_wait(&full[s], mpar)) {
          fail(kErrTimeoutFull);
          stop = true;
          break;
        }
        if (++ms == stages) {
          ms = 0;
          mpar ^= 1u;
        }
        // AMN: [M half][piece][32 K rows][128 bytes]; else [piece][128 rows][64 bytes]
        constexpr uint64_t apiece = (AMN ? kTpBK * 128 : kTpPieceA) >> 4, akstep = AMN ? 128 : 2;
        constexpr uint64_t bpiece = Cfg::PIECE_B >> 4;
        const uint64_t da = dA0 + (uint64_t)((s * Cfg::STAGE) >> 4), db = dB0 + (uint64_t)((s * Cfg::STAGE) >> 4);
#pragma unroll
        for (int kk = 0; kk < kTpBK / 16; ++kk) {
          const uint64_t a0 = da + kk * akstep, a1 = a0 + apiece, a2 = a1 + apiece;
          const uint64_t b0 = db + kk * 2, b1 = b0 + bpiece, b2 = b1 + bpiece;
          mma_bf16<kColNone>(dt, a2, b0, idesc, kb != w.kb0 || kk != 0);
          mma_bf16<kColFill>(dt, a1, b1, idesc, 1);
          mma_bf16<kColLast>(dt, a1, b0, idesc, 1);
          mma_bf16<kColFill>(dt, a0, b2, idesc, 1);
          mma_bf16<kColUse>(dt, a0, b1, idesc, 1);
          mma_bf16<kColLast>(dt, a0, b0, idesc, 1);
        }
        mma_commit(&empty[s]);
      }
      if (stop) break;
      mma_commit(&acc_full[slot]);
    }
    mma_commit(&drain);
    mbar_wait(&drain, 0);
  } else if (warp == 2 && lane == 0) {
    // ---------------- publishes the x1 tiles of a two-pass launch: waits for
    // the epilogue warps' stores to be issued, then releases the counters of
    // the tile's slabs (the release is cumulative over those stores)
    for (uint32_t k = 0;; ++k) {
      const TpUnit w = next_unit(k);
      if (!w.d) break;
      if (!dynamic) continue;
      if (!mbar_wait(&stored[k & 1], (k >> 1) & 1)) {
        fail(kErrTimeoutDone);
        break;
      }
      mbar_arrive(&acc_empty[k & 1]);  // keeps the epilogue within two units of this thread
      if (w.pass == 0) {
        const TpPass* d = w.d;
        const int s0 = d->slabs > 1 ? w.mt * kBM / d->R : 0;
        const int s1 = d->slabs > 1 ? (min((w.mt + 1) * kBM, d->M) - 1) / d->R : 0;
        for (int s = s0; s <= s1; ++s)
          red_release(d->dep + (w.c * d->slabs + s) * d->dep_tn + (d->dep_tn > 1 ? w.nt : 0), 1u);
      }
    }
  } else if (warp >= 4) {
    // ---------------- epilogue
    pdl_wait();
    const int q = warp & 3, cg = ((warp - 4) >> 2) & 1, slot = (warp - 4) / kTpEpi;
    auto lane_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      if (__all_sync(0xffffffffu, mbar_wait(bar, parity))) return true;
      if (lane == 0) fail(kErrTimeoutDone);
      return false;
    };
    auto arrive = [&](uint64_t* bar) {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    };
    for (uint32_t k = slot;; k += 2) {
      const int sl = k % kTpSched;
      if (!lane_wait(&sched_full[sl], (k / kTpSched) & 1)) break;
      const TpUnit w = sched_unit[sl];
      arrive(&sched_empty[sl]);
      if (!w.d) break;
      const TpPass* D = w.d;
      const int c = w.c;
      const int M = D->M, N = D->N, R = D->R, n0 = w.nt * w.bn;
      const int ncols = min(w.bn, N - n0);           // columns with output (a multiple of 8)
      const int m = w.mt * kBM + q * 32 + lane;
      const bool mrow = m < M;
      const int sb = D->slabs > 1 ? m / R : 0;       // slab of this row
      const int64_t off = (int64_t)sb * R * N + (m - sb * R) + (int64_t)n0 * R;
      const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(slot * 256);
      const bool pieces = D->outp[c] != nullptr;
      const int ncol = mrow ? N - n0 : 0;            // columns this lane may touch
      if (pieces) {
        // lanes pair up (rows m, m + 1 of one slab: R is even): of two columns
        // the even lane takes the first and the odd lane the second, each with
        // both rows, so every store writes two values of one piece (4 bytes)
        const bool odd = lane & 1;
        const int64_t plane2 = (int64_t)M * N / 2;
        uint32_t* op = reinterpret_cast<uint32_t*>(D->outp[c]) + ((off + (odd ? R - 1 : 0)) >> 1);
        if (!lane_wait(&acc_full[slot], (k >> 1) & 1)) break;
        tc_fence_after();
        for (int col0 = cg * 8; col0 < ncols; col0 += 16) {
          uint32_t r[8];
          tp_ld(ta + (uint32_t)col0, r);
          tmem_wait_ld();
          tp_fence(r);
          uint32_t* o = op + (int64_t)(col0 >> 1) * R;
#pragma unroll
          for (int j = 0; j < 8; j += 2, o += R) {
            const float x0 = __uint_as_float(r[j]), x1 = __uint_as_float(r[j + 1]);
            const float got = __shfl_xor_sync(0xffffffffu, odd ? x0 : x1, 1);
            if (col0 + j < ncol) {  // (N is even: both columns of a pair exist)
              uint32_t p0, p1, p2;
              split3_pair(odd ? got : x0, odd ? x1 : got, p0, p1, p2);
              o[0] = p0;
              o[plane2] = p1;
              o[2 * plane2] = p2;
            }
          }
        }
      } else {
        // out = base + alpha acc (EPI 1, 2: compensated state and indicators).
        // The inputs of a chunk are loaded before its accumulator is read, the
        // first ones before it is complete.
        constexpr int W = 8;
        const float sc = D->alpha;
        const float* bsrc = D->base[c] ? D->base[c] + off : nullptr;
        float* of = D->outf[c] + off;
        float* lp = (EPI > 0 && D->lo[c]) ? D->lo[c] + off : nullptr;
        double* ind = nullptr;
        if (EPI == 2 && D->ind) ind = D->ind + 4 * (__ldcg(D->ind_ctr) % D->ind_k) + c;
        IndSums sums;
        float bb[W], lv[EPI > 0 ? W : 1], pv[EPI == 2 ? W : 1];
        auto load_in = [&](int col0) {
#pragma unroll
          for (int j = 0; j < W; ++j) {
            const bool ok = col0 + j < ncol;
            const int64_t o = (int64_t)(col0 + j) * R;
            bb[j] = (ok && bsrc) ? __ldg(bsrc + o) : 0.f;
            if constexpr (EPI > 0) lv[j] = (ok && lp) ? __ldcg(lp + o) : 0.f;
            if constexpr (EPI == 2) pv[j] = (ok && ind) ? __ldcg(of + o) : 0.f;
          }
        };
        load_in(cg * 8);
        if (!lane_wait(&acc_full[slot], (k >> 1) & 1)) break;
        tc_fence_after();
        for (int col0 = cg * 8; col0 < ncols; col0 += 16) {
          {
            uint32_t r[W];
            tp_ld(ta + (uint32_t)col0, r);
            tmem_wait_ld();
            tp_fence(r);
            float hi[W], lo[EPI > 0 ? W : 1];
#pragma unroll
            for (int j = 0; j < W; ++j) {
              const float a = __uint_as_float(r[j]);
              if constexpr (EPI == 0) {
                hi[j] = __fmaf_rn(sc, a, bb[j]);
              } else {
                if (lp) {
                  comp_update(bb[j], lv[j], __fmul_rn(sc, a), hi[j], lo[j]);
                } else {
                  hi[j] = __fmaf_rn(sc, a, bb[j]);
                  lo[j] = 0.f;
                }
              }
              if constexpr (EPI == 2) {
                const int col = n0 + col0 + j;
                if (ind && col0 + j < ncol) sums.add(hi[j], pv[j], col == 0 || col == N - 1);
              }
            }
            if (col0 + 16 < ncols) load_in(col0 + 16);
#pragma unroll
            for (int j = 0; j < W; ++j)
              if (col0 + j < ncol) {
                const int64_t o = (int64_t)(col0 + j) * R;
                of[o] = hi[j];
                if constexpr (EPI > 0) {
                  if (lp) lp[o] = lo[j];
                }
              }
          }
        }
        if constexpr (EPI == 2) {
          if (ind) {
            double wm = 0.0;  // trapezoid weight of row m
            if (mrow)
              wm = D->ind_n2 > 0 ? trap_w(m % D->ind_n1, D->ind_n1) * trap_w(m / D->ind_n1, D->ind_n2)
                                 : trap_w(m, D->ind_n1);
            sums.flush(wm, ind);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&acc_empty[slot]);  // every column of this slot has been read
        if (dynamic) mbar_arrive(&stored[slot]);
      }
      if (__any_sync(0xffffffffu, *abort_v)) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (dynamic && L.clear) {
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(L.ctl + 1, 1u) == gridDim.x - 1) {
        __threadfence();
        abort_flag = 2;
      }
    }
    __syncthreads();
    if (abort_flag == 2)
      for (int i = threadIdx.x; i < L.nctl; i += blockDim.x) L.ctl[i] = 0u;
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ---------------------------------------------------------------- pointwise
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// 3D stencil and reaction for rows of up to 192 points.  A block owns 8 rows
// (y0 .. y0 + 7), one per warp, and marches zlen planes.  Each plane of u and
// v (its 8 rows and the two beside them) arrives by one TMA copy per field
// into a ring of shared-memory slots; a row's own values stay in registers
// for the next two planes, where they are the z neighbours.  The warps wait
// for a plane and release its slot each on its own, without a barrier of the
// block per plane; the first one issues the copies.  NSEG = 64-point segments
// of a row, two points a lane: sides such as 64, 96, 160 and 192 leave fewer
// lanes idle than four points a lane would.
constexpr int kRowRingY = 8;
static_assert(kRowRingY == kPwWarps, "one row per warp");
constexpr int kRowRingX = 192;
constexpr int kRowRingField = kRowRingX * (kRowRingY + 2);   // floats per field and plane
constexpr int kRowRingSlots = 5;
constexpr int kRowRingSmem = kRowRingSlots * 2 * kRowRingField * 4 + 128 + 2 * kRowRingSlots * 8;
// The x direction at point j of a pair starting at an even index, on a row of
// even length: only j = 0 can be the first point and only j = 1 the last.
__device__ __forceinline__ float tri_x2(int j, float xm, float xc, float xp, int i, int n, float lo,
                                        float up, float b0, float bn) {
  if (j == 0 && i == 0) return b0 * (xp - xc);
  if (j == 1 && i == n - 1) return bn * (xm - xc);
  return tri_in(xm, xc, xp, lo, up);
}
__device__ __forceinline__ dfloat dtri_x2(int j, float xm, float xc, float xp, int i, int n,
                                          const CoefDF& c) {
  if (j == 0 && i == 0) return c.b0 * df_diff(xp, xc);
  if (j == 1 && i == n - 1) return c.bn * df_diff(xm, xc);
  return dtri_in(xm, xc, xp, c.lo, c.up);
}
template <int NSEG, bool DF>
__global__ void __launch_bounds__(kPwThreads, 2) rhs3_row_kernel(const __grid_constant__ PwLaunch L) {
  extern __shared__ uint8_t smem_raw[];
  float* ring = (float*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
  uint64_t* full = (uint64_t*)(ring + kRowRingSlots * 2 * kRowRingField);
  uint64_t* empty = full + kRowRingSlots;
  __shared__ PwDesc sd;
  int lb;
  const PwDesc* home = nullptr;
  const PwDesc* dp = block_desc(L, &sd, lb, &home);
  indicator_open_step(dp, lb);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nx = dp->nx, ny = dp->ny, nz = dp->nz;
  const int ytiles = (ny + kRowRingY - 1) / kRowRingY;
  const int y0 = (lb % ytiles) * kRowRingY;
  const int z0 = (lb / ytiles) * dp->zlen, z1 = min(z0 + dp->zlen, nz);
  const int plo = max(z0 - 1, 0), phi = min(z1, nz - 1);
  const int np = phi - plo + 1;
  const CUtensorMap* mu = &home->tu;
  const CUtensorMap* mv = &home->tv;
  const uint32_t tx = (uint32_t)(2 * nx * (kRowRingY + 2) * 4);
  if (threadIdx.x == 0) {
    for (int sl = 0; sl < kRowRingSlots; ++sl) {
      mbar_init(&full[sl], 1);
      mbar_init(&empty[sl], kRowRingY);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // copies (one thread): every plane whose slot is free, and planes up to
  // `need` in any case
  int issued = 0;
  auto issue = [&](int need) -> bool {
    for (; issued < np; ++issued) {
      const int sl = issued % kRowRingSlots;
      if (issued >= kRowRingSlots) {
        const uint32_t par = (uint32_t)(issued / kRowRingSlots - 1) & 1u;
        if (issued < need ? !mbar_wait(&empty[sl], par) : !mbar_test_wait(&empty[sl], par)) return issued >= need;
      }
      float* dst = ring + sl * 2 * kRowRingField;
      mbar_arrive_expect_tx(&full[sl], tx);
      tma_load_3d(dst, mu, &full[sl], 0, y0 - 1, plo + issued);
      tma_load_3d(dst + kRowRingField, mv, &full[sl], 0, y0 - 1, plo + issued);
    }
    return true;
  };
  const ReactionT<float>& rx = dp->a.rx;
  const int64_t N = dp->a.N;
  uint32_t* ou = reinterpret_cast<uint32_t*>(dp->wu);  // two values of a piece a word
  uint32_t* ov = reinterpret_cast<uint32_t*>(dp->wv);
  const int y = y0 + warp;
  const bool rowok = y < ny;
  const int o0 = (warp + 1) * nx;
  float2 um[NSEG], vm[NSEG], uc[NSEG], vc[NSEG];  // planes z - 1 and z of this row
  int got = 0;           // planes known to have landed
  bool lost = false;
  auto arrive = [&](int q) {  // this warp is done with plane plo + q
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[q % kRowRingSlots]);
  };
  for (int z = z0; z < z1 && !lost; ++z) {
    const int need = min(z + 1, phi) - plo + 1;  // planes z - 1 .. z + 1
    if (threadIdx.x == 0) issue(need);
    for (; got < need && !lost; ++got)
      lost = !__all_sync(0xffffffffu,
                         mbar_wait(&full[got % kRowRingSlots], (uint32_t)(got / kRowRingSlots) & 1u));
    if (lost) {
      if (lane == 0) atomicCAS(L.err, 0, kErrTimeoutFull);
      break;
    }
    if (!rowok) {
      if (z == z0 && z0 > plo) arrive(0);
      arrive(z - plo);
      continue;
    }
    const float* pc = ring + ((z - plo) % kRowRingSlots) * 2 * kRowRingField;
    const float* pp = z + 1 < nz ? ring + ((z + 1 - plo) % kRowRingSlots) * 2 * kRowRingField : nullptr;
    if (z == z0) {
      const float* pm = z > 0 ? ring + ((z - 1 - plo) % kRowRingSlots) * 2 * kRowRingField : pc;
#pragma unroll
      for (int s = 0; s < NSEG; ++s) {
        const int x = 64 * s + 2 * lane;
        const bool a = x < nx;
        um[s] = a ? *reinterpret_cast<const float2*>(pm + o0 + x) : make_float2(0.f, 0.f);
        vm[s] = a ? *reinterpret_cast<const float2*>(pm + kRowRingField + o0 + x) : make_float2(0.f, 0.f);
        uc[s] = a ? *reinterpret_cast<const float2*>(pc + o0 + x) : make_float2(0.f, 0.f);
        vc[s] = a ? *reinterpret_cast<const float2*>(pc + kRowRingField + o0 + x) : make_float2(0.f, 0.f);
      }
    }
    const bool yin = y > 0 && y + 1 < ny, zin = z > 0 && z + 1 < nz;  // uniform over the warp
    constexpr int NP = 2 * NSEG;
    float cu[NP], cv[NP], wu[NP], wv[NP];
    dfloat du[DF ? NP : 1], dv[DF ? NP : 1];
    const TridiagT<float>(&A)[2][3] = dp->a.A;
    const TridiagT<float>(&Al)[2][3] = dp->a.Alo;
#pragma unroll
    for (int s = 0; s < NSEG; ++s) {
      const int x = 64 * s + 2 * lane;
      const int o = o0 + (x < nx ? x : 0);
      const float* pv = pc + kRowRingField;
      const float2 uym = *reinterpret_cast<const float2*>(pc + o - nx);
      const float2 vym = *reinterpret_cast<const float2*>(pv + o - nx);
      const float2 uyp = *reinterpret_cast<const float2*>(pc + o + nx);
      const float2 vyp = *reinterpret_cast<const float2*>(pv + o + nx);
      const float2 uzp = pp ? *reinterpret_cast<const float2*>(pp + o) : make_float2(0.f, 0.f);
      const float2 vzp = pp ? *reinterpret_cast<const float2*>(pp + kRowRingField + o) : make_float2(0.f, 0.f);
      const float ul = pc[o - 1], vl = pv[o - 1];            // x = 0: the row before's last value, unused
      const float ur = pc[o + 2], vr = pv[o + 2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i = 2 * s + j, xi = x + j;
        cu[i] = j ? uc[s].y : uc[s].x;
        cv[i] = j ? vc[s].y : vc[s].x;
        const float lu = j ? uc[s].x : ul, lv = j ? vc[s].x : vl;
        const float ru = j ? ur : uc[s].y, rv = j ? vr : vc[s].y;
        const float um_ = j ? um[s].y : um[s].x, vm_ = j ? vm[s].y : vm[s].x;
        const float up_ = j ? uzp.y : uzp.x, vp_ = j ? vzp.y : vzp.x;
        const float uy0 = j ? uym.y : uym.x, uy1 = j ? uyp.y : uyp.x;
        const float vy0 = j ? vym.y : vym.x, vy1 = j ? vyp.y : vyp.x;
        if constexpr (DF) {  // accurate mode: stencil and reaction in double-float, one rounding
          const CoefDF dxu = coef_df(A[0][0], Al[0][0]), dxv = coef_df(A[1][0], Al[1][0]);
          const CoefDF dyu = coef_df(A[0][1], Al[0][1]), dyv = coef_df(A[1][1], Al[1][1]);
          const CoefDF dzu = coef_df(A[0][2], Al[0][2]), dzv = coef_df(A[1][2], Al[1][2]);
          du[i] = dtri_x2(j, lu, cu[i], ru, xi, nx, dxu) +
                  dtri_dir(uy0, cu[i], uy1, y, ny, dyu.lo, dyu.up, dyu.b0, dyu.bn) +
                  dtri_dir(um_, cu[i], up_, z, nz, dzu.lo, dzu.up, dzu.b0, dzu.bn);
          dv[i] = dtri_x2(j, lv, cv[i], rv, xi, nx, dxv) +
                  dtri_dir(vy0, cv[i], vy1, y, ny, dyv.lo, dyv.up, dyv.b0, dyv.bn) +
                  dtri_dir(vm_, cv[i], vp_, z, nz, dzv.lo, dzv.up, dzv.b0, dzv.bn);
        } else {
          float ku = tri_x2(j, lu, cu[i], ru, xi, nx, A[0][0].lo, A[0][0].up, A[0][0].b0, A[0][0].bn);
          float kv = tri_x2(j, lv, cv[i], rv, xi, nx, A[1][0].lo, A[1][0].up, A[1][0].b0, A[1][0].bn);
          if (yin && zin) {
            ku += tri_in(uy0, cu[i], uy1, A[0][1].lo, A[0][1].up);
            kv += tri_in(vy0, cv[i], vy1, A[1][1].lo, A[1][1].up);
            ku += tri_in(um_, cu[i], up_, A[0][2].lo, A[0][2].up);
            kv += tri_in(vm_, cv[i], vp_, A[1][2].lo, A[1][2].up);
          } else {
            ku += tri_dir(uy0, cu[i], uy1, y, ny, A[0][1].lo, A[0][1].up, A[0][1].b0, A[0][1].bn);
            kv += tri_dir(vy0, cv[i], vy1, y, ny, A[1][1].lo, A[1][1].up, A[1][1].b0, A[1][1].bn);
            ku += tri_dir(um_, cu[i], up_, z, nz, A[0][2].lo, A[0][2].up, A[0][2].b0, A[0][2].bn);
            kv += tri_dir(vm_, cv[i], vp_, z, nz, A[1][2].lo, A[1][2].up, A[1][2].b0, A[1][2].bn);
          }
          wu[i] = ku;
          wv[i] = kv;
        }
      }
      um[s] = uc[s];
      vm[s] = vc[s];
      uc[s] = uzp;
      vc[s] = vzp;
    }
    // plane z - 1 has been read (in the first iteration), and so has plane z:
    // what the next planes need of it is in registers
    if (z == z0 && z0 > plo) arrive(0);
    arrive(z - plo);
    for_model<NP>(rx, [&](const ReactionT<float>& r, int i) {
      if constexpr (DF) {
        dfloat gu, gv;
        react_dfd(r, cu[i], cv[i], gu, gv);
        wu[i] = df_round(du[i] + gu);
        wv[i] = df_round(dv[i] + gv);
      } else {
        float gu, gv;
        react<float>(r, cu[i], cv[i], gu, gv);
        wu[i] += gu;
        wv[i] += gv;
      }
    });
    const int64_t row = ((int64_t)z * ny + y) * nx;
#pragma unroll
    for (int s = 0; s < NSEG; ++s) {
      const int x = 64 * s + 2 * lane;
      if (x < nx) {
        const int64_t i2 = (row + x) >> 1;
        uint32_t p0, p1, p2;
        split3_pair(wu[2 * s], wu[2 * s + 1], p0, p1, p2);
        ou[i2] = p0;
        ou[N / 2 + i2] = p1;
        ou[N + i2] = p2;
        split3_pair(wv[2 * s], wv[2 * s + 1], p0, p1, p2);
        ov[i2] = p0;
        ov[N / 2 + i2] = p1;
        ov[N + i2] = p2;
      }
    }
  }
  // every copy has landed before the block's shared memory is released
  if (threadIdx.x == 0)
    for (int q = max(0, issued - kRowRingSlots); q < issued; ++q)
      mbar_wait(&full[q % kRowRingSlots], (uint32_t)(q / kRowRingSlots) & 1u);
}
