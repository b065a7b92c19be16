// Block walk for D = 64 (included by la_tc.cu, inside its anonymous namespace, after the helpers).
//
// One thread block walks the 128-token blocks of one (batch*head, segment), 64 features by 64 value columns.  Per block
// (i, j: tokens, d: features, e: value columns)
//   M1  S       [i, j] = a b^T                    A, B in shared memory, K = 64
//   M2  O_inter [i, e] = a Z_hi (+ a Z_lo + a Y)  A, B in shared memory, K = 64
//   M3  dZ^T    [(e, e), d] = [fc_hi | fc_lo]^T b  A in tensor memory, K = 128     (fc = diag(f_state) c)
//   M4  O_intra [i, e] = P_hi c (+ P_lo c)        A = P in tensor memory, in the place of S, K = 128
// and the CUDA cores form P = S (.) D, out = O_intra + diag(f_out) O_inter and Z <- Gamma Z + dZ.
// An instruction has 128 rows whatever D is, so M3 puts the hi terms of fc in one half of the lanes and the lo terms in the
// other: one product of half the columns for both.  Its two halves stay apart: Z is the state that the hi terms add up to, Y the one of
// the lo terms, 2^-9 of it, for which one bf16 operand is as good as two for Z.  They meet in M2, and in the state that is handed
// out.
//
// The only chain between blocks is Z in registers.  The walk before this one (products of zero-padded rows, fc made between dZ and
// the next state operand by the same warps, each waiting for the other) took 2.5 us a block.  The products of iteration n are M1(n+1)
// M2(n) M4(n) M3(n+1), 1900 clocks, and each operand is made while others run: S(n+1) has until M4 of the next iteration, dZ(n) and
// fc(n+1) have M1, M2 and M4, the accumulators of M4(n) are read during M3(n+1) and M1(n+2), the state operand is written after M2(n).
// A block takes 4000 to 4400 clocks where memory is not the bound (one thread block per SM, HBM: 3500 at fp32 results): the state
// group's dZ (350), fc (2000, sharing the schedulers with scores and output) and operand (500), and M3, come one after the other.
// Measured, us, before and after: 2 x 16 heads x 8192, fp32 results, forward 68 and 50, backward 162 and 130; 1 x 32 x 16384 117 and 92,
// 285 and 241.
//
// Tensor memory (512 columns): S/P 2 x 128, O_inter 64, O_intra 64, dZ 64, fc 64.
// Shared memory: three stages of a, b, c (48 KB each), the state operand (Z hi, Z lo, Y: 8 KB each), the output on its way to
// its bulk store (16 or 32 KB).
// Warp roles (28 warps): 0 TMA producer, 1 MMA issuer (converged), 4-11 P, 12-19 state and fc (quarters 0, 1 of tensor memory:
// hi terms and Z, quarters 2, 3: lo terms and Y; forward the other way round), 20-27 output.
//
// Packed batch: the rows past a sequence's end are its neighbour's.  Their scores are masked and their outputs not stored; so
// that their values cannot come through a zero weight either (0 * inf), the state group clears those rows of b and c before M3.

constexpr int V_THREADS = 896;
constexpr int V_STAGES = 3;
constexpr uint32_t VCOL_S = 0, VCOL_OE = 256, VCOL_OI = 320, VCOL_DZ = 384, VCOL_F = 448;
constexpr int V_REGS_LAUNCH = 72, V_REGS_CTL = 24, V_REGS_P = 64, V_REGS_Z = 96, V_REGS_O = 80;
static_assert(4 * V_REGS_CTL + 8 * (V_REGS_P + V_REGS_Z + V_REGS_O) <= 28 * V_REGS_LAUNCH, "registers of the launch");

enum VBar {
  V_FULL_AB0 = 0,                    // TMA -> MMA: a and b of a stage
  V_FULL_C0 = V_FULL_AB0 + V_STAGES, // TMA -> state group, MMA: c
  V_FREE0 = V_FULL_C0 + V_STAGES,    // M4 done: the stage may be loaded again
  V_S_READY0 = V_FREE0 + V_STAGES, V_S_READY1,  // M1 of an even / odd block done
  V_P_READY0, V_P_READY1,            // P written (8 warps)
  V_Z_READY,                         // state operand written (8 warps)
  V_FC_READY,                        // fc written and the dZ before it read (8 warps)
  V_M2_DONE,                         // the state operand may be written
  V_DZ_READY,                        // M3 done: dZ complete, fc free
  V_O_READY,                         // M4 done: both accumulators complete
  V_O_FREE,                          // both accumulators read (8 warps)
  V_STAGED,                          // output rows in shared memory (8 warps)
  V_STORED,                          // ... and read by their bulk store
  V_FINAL,                           // the lo half of the state that is handed out (4 warps)
  V_DRAIN,
  V_NUM_BARS
};

template <typename TOut>
struct alignas(1024) VSmem {
  struct Stage {
    __nv_bfloat16 a[128 * 64], b[128 * 64], c[128 * 64];
  } st[V_STAGES];
  __nv_bfloat16 z[3][64 * 64];  // Z hi, Z lo, Y: [e][d]
  unsigned char out[sizeof(TOut) / 2][128 * 128];
  float gseg[3];   // decay through a whole segment, through the sequence's last one, and through all before this one
  uint64_t bars[V_NUM_BARS];
  uint32_t tmem_slot;
  int abort;
};

// Maps over the outputs of both jobs, and over the second half of the first one's (OpArgs::out2).
struct VOutMaps {
  CUtensorMap of[2], second_half;
};

// args.njobs == 2: see tc_walk_kernel.
template <bool REV, typename TOut>
__global__ void __launch_bounds__(V_THREADS, 1)
tc_walk64_kernel(const __grid_constant__ TcMaps maps0, const __grid_constant__ TcMaps maps1, const __grid_constant__ VOutMaps maps_out,
                 const __grid_constant__ TcArgs args, const __grid_constant__ DecayTable tab) {
  extern __shared__ unsigned char smem_raw[];
  using Sm = VSmem<TOut>;
  Sm& sm = *reinterpret_cast<Sm*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (args.follows == FOLLOWS_ANY && args.seq_start) grid_dep_wait();  // the tables of a packed batch
  const int jobid = (args.njobs == 2) ? (int)(blockIdx.x & 1) : 0;
  const int bidx = (args.njobs == 2) ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const TcJob& job = args.job[jobid];
  const TcMaps* const maps = jobid ? &maps1 : &maps0;
  const int seg = bidx % args.nseg;
  int bh = bidx / args.nseg;
  if (args.seq_order) bh = args.seq_order[bh / args.H] * args.H + bh % args.H;
  const int hh_ = bh % args.H;
  const int n_tok = args.seq_len ? args.seq_len[bh / args.H] : args.N;
  const int tok0 = args.seq_start ? args.seq_start[bh / args.H] : 0;
  const int nseg_own = (n_tok + args.seg_len - 1) / args.seg_len;
  if (seg >= nseg_own) return;  // the grid covers the longest sequence; nothing has been set up yet
  const int seg_t0 = seg * args.seg_len;
  const int seg_t1 = min(n_tok, seg_t0 + args.seg_len);
  const int nblk = (seg_t1 - seg_t0 + 127) >> 7;
  const int edge_len = seg_t1 - seg_t0 - (nblk - 1) * 128;  // tokens of the block that holds the segment's last ones
  const bool shared_tail = args.seq_start && edge_len < 128;
  const float s2 = (float)tab.s2[hh_];
  const int before = REV ? nseg_own - 1 - seg : seg;  // segments walked before this one
  const bool has_entry = job.z_in != nullptr || before > 0;  // else the first block has no O_inter: M2 is skipped
  const bool want_final = job.final_out && (REV ? seg == 0 : seg == nseg_own - 1);
  // (a shared tail: for the rows that are cleared before it)
  const bool last_m3 = want_final || (shared_tail && (!REV || nblk == 1));
  const bool split_p = (args.precision & 1) != 0, split_z = (args.precision & 2) != 0;
  const bool split_c = (args.precision & 4) != 0 && s2 != 0.f;  // lambda == 1: the lo terms are identically zero
  const int bb_ = args.seq_start ? 0 : bh / args.H;

  if (tid == 0) {
    for (int i = 0; i < V_NUM_BARS; ++i) {
      uint32_t count = 1;
      if (i == V_P_READY0 || i == V_P_READY1 || i == V_Z_READY || i == V_FC_READY || i == V_O_FREE || i == V_STAGED) count = 8;
      if (i == V_FINAL) count = 4;
      mbar_init(&sm.bars[i], count);
    }
    sm.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    if (args.follows == FOLLOWS_ANY) grid_dep_wait();  // (see Follows)
    tmem_alloc(&sm.tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  if (warp == 4 && lane < 3) {
    const int len = lane == 0 ? args.seg_len : lane == 1 ? n_tok - (nseg_own - 1) * args.seg_len : REV ? n_tok - seg_t1 : seg_t0;
    sm.gseg[lane] = decay_pow_d(tab.s2[hh_], (double)len);
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sm.tmem_slot;
  if (args.follows == FOLLOWS_ANY) {
    grid_dep_wait();
    grid_dep_launch();
  }

  if (warp < 4) {
    set_regs<V_REGS_CTL, V_REGS_LAUNCH>();
    if (warp == 0) {
      // ------------------------------------ TMA producer ------------------------------------
      if (lane == 0) {
        const int bf_ = args.fold && bb_ >= args.fold ? bb_ - args.fold : bb_;  // of an operand that is shared
        const int ba = job.shared & SHARED_A ? bf_ : bb_, bb = job.shared & SHARED_B ? bf_ : bb_, bc = job.shared & SHARED_C ? bf_ : bb_;
        int armed = 0;  // blocks whose loads have been started
        for (int it = 0, s = 0, phase = 0; it < nblk; ++it) {
          if (it >= V_STAGES) TC_WAIT_TO(producer_done, V_FREE0 + s, phase ^ 1, 1);
          const int t = tok0 + seg_t0 + (REV ? (nblk - 1 - it) : it) * 128;
          mbar_arrive_expect_tx(&sm.bars[V_FULL_AB0 + s], 32768);
          tma_load_4d(sm.st[s].b, &maps->b, &sm.bars[V_FULL_AB0 + s], 0, t, hh_, bb);
          tma_load_4d(sm.st[s].a, &maps->a, &sm.bars[V_FULL_AB0 + s], 0, t, hh_, ba);
          mbar_arrive_expect_tx(&sm.bars[V_FULL_C0 + s], 16384);
          tma_load_4d(sm.st[s].c, &maps->c, &sm.bars[V_FULL_C0 + s], 0, t, hh_, bc);
          armed = it + 1;
          if (++s == V_STAGES) s = 0, phase ^= 1;
        }
      producer_done:
        if (sm.abort) {  // nothing may be in flight when the block exits
          for (int k = 0; k < V_STAGES; ++k) {
            const int b = armed - 1 - k;
            if (b < 0) break;
            drain_wait(&sm.bars[V_FULL_AB0 + b % V_STAGES], (b / V_STAGES) & 1);
            drain_wait(&sm.bars[V_FULL_C0 + b % V_STAGES], (b / V_STAGES) & 1);
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------ MMA issuer ------------------------------------
      constexpr uint32_t ID_S = umma_idesc_bf16(128, 128, false, false);
      constexpr uint32_t ID_KK = umma_idesc_bf16(128, 64, false, false);  // K-major B
      constexpr uint32_t ID_KN = umma_idesc_bf16(128, 64, false, true);   // MN-major B
      constexpr uint32_t HI = UMMA_DESC_HI_SBO1024;
      constexpr uint32_t KMAJ = 1u << 16, MNMAJ = 1024u << 16;  // leading-dimension offset 16 bytes / 16 KB (one panel: unused)
      const uint32_t go = elect_one();
      const uint32_t base = (smem_u32(&sm) & 0x3FFFFu) >> 4;
      constexpr uint32_t OA = (uint32_t)(offsetof(typename Sm::Stage, a) >> 4), OB = (uint32_t)(offsetof(typename Sm::Stage, b) >> 4);
      constexpr uint32_t OC = (uint32_t)(offsetof(typename Sm::Stage, c) >> 4), STAGE = (uint32_t)(sizeof(typename Sm::Stage) >> 4);
      constexpr uint32_t OZ = (uint32_t)(offsetof(Sm, z) >> 4) + KMAJ, ZTILE = 512;
      uint32_t s = 0, phase = 0;  // the present block's stage
      TC_WAIT_WARP_TO(mma_done, V_FULL_AB0, 0, 7);
      tc_fence_after_sync();
      umma_group_ss<4, true, true>(tmem + VCOL_S, base + OA + KMAJ, base + OB + KMAJ, HI, ID_S, 0, go);
      umma_commit_if(&sm.bars[V_S_READY0], go);
      if (nblk > 1 || last_m3) {
        TC_WAIT_WARP_TO(mma_done, V_FC_READY, 0, 13);
        tc_fence_after_sync();
        umma_group_tsd<false>(tmem + VCOL_DZ, tmem + VCOL_F, base + OB + MNMAJ, HI, ID_KN, 0, go);
        umma_commit_if(&sm.bars[V_DZ_READY], go);
      }
      for (int it = 0; it < nblk; ++it) {
        const uint32_t par = it & 1;
        const uint32_t buf = base + s * STAGE;
        const uint32_t s1 = s + 1 == V_STAGES ? 0 : s + 1, phase1 = s + 1 == V_STAGES ? phase ^ 1 : phase;
        const uint32_t buf1 = base + s1 * STAGE;
        const bool more = it + 1 < nblk;
        if (more) {
          TC_WAIT_WARP_TO(mma_done, V_FULL_AB0 + s1, phase1, 11);
          tc_fence_after_sync();
          umma_group_ss<4, true, true>(tmem + VCOL_S + (par ^ 1) * 128, buf1 + OA + KMAJ, buf1 + OB + KMAJ, HI, ID_S, 0, go);
          umma_commit_if(&sm.bars[V_S_READY0 + (par ^ 1)], go);
        }
        TC_WAIT_WARP_TO(mma_done, V_Z_READY, par, 12);
        if (it > 0) TC_WAIT_WARP_TO(mma_done, V_O_FREE, par ^ 1, 16);
        tc_fence_after_sync();
        if (it > 0 || has_entry) {
          umma_group_ss<4, true, true>(tmem + VCOL_OE, buf + OA + KMAJ, base + OZ, HI, ID_KK, 0, go);
          if (split_z) umma_group_ss<4, true, true>(tmem + VCOL_OE, buf + OA + KMAJ, base + OZ + ZTILE, HI, ID_KK, 1, go);
          if (split_c && it > 0) umma_group_ss<4, true, true>(tmem + VCOL_OE, buf + OA + KMAJ, base + OZ + 2 * ZTILE, HI, ID_KK, 1, go);
        }
        umma_commit_if(&sm.bars[V_M2_DONE], go);
        TC_WAIT_WARP_TO(mma_done, V_FULL_C0 + s, phase, 15);
        TC_WAIT_WARP_TO(mma_done, V_P_READY0 + par, (it >> 1) & 1, 14);
        tc_fence_after_sync();
        const uint32_t col_p = tmem + VCOL_S + par * 128;
        umma_group_ts8(tmem + VCOL_OI, col_p, buf + OC + MNMAJ, HI, ID_KN, 0, go);
        if (split_p) umma_group_ts8(tmem + VCOL_OI, col_p + 8, buf + OC + MNMAJ, HI, ID_KN, 1, go);
        umma_commit_if(&sm.bars[V_O_READY], go);
        umma_commit_if(&sm.bars[V_FREE0 + s], go);
        if (more && (it + 2 < nblk || last_m3)) {
          TC_WAIT_WARP_TO(mma_done, V_FC_READY, par ^ 1, 13);
          tc_fence_after_sync();
          umma_group_tsd<false>(tmem + VCOL_DZ, tmem + VCOL_F, buf1 + OB + MNMAJ, HI, ID_KN, 0, go);
          umma_commit_if(&sm.bars[V_DZ_READY], go);
        }
        s = s1;
        phase = phase1;
      }
    mma_done:
      if (sm.abort) {
        umma_commit_if(&sm.bars[V_DRAIN], go);
        drain_wait(&sm.bars[V_DRAIN], 0);
      }
    }
  } else if (warp < 12) {
    // ------------------------------------ P: S -> masked, decayed bf16 hi / lo in its place ------------------------------------
    set_regs<V_REGS_P, V_REGS_LAUNCH>();
    const int q = warp & 3, half = (warp - 4) >> 2;  // score rows q * 32 + lane, keys half * 64 .. + 63
    const int r = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    // (reverse walk of a packed batch: the keys past the end of the sequence lie inside the band of the edge block)
    const int cut = REV && args.seq_start ? edge_len : 128;
    const float lam1 = ex2_approx(-s2), lam2 = ex2_approx(-s2 * 2.f), lam4 = ex2_approx(-s2 * 4.f), lam8 = ex2_approx(-s2 * 8.f);
    for (int it = 0; it < nblk; ++it) {
      const int s = it & 1;
      const uint32_t colS = lane_addr + VCOL_S + s * 128;
      const bool edge = REV && it == 0 && cut < 128;
      TC_WAIT_WARP(V_S_READY0 + s, (it >> 1) & 1, 17);
      tc_fence_after_sync();
#pragma unroll 1
      for (int pi = 0; pi < 4; ++pi) {
        const int j0 = half * 64 + pi * 16;
        const int off = REV ? q - (j0 >> 5) : (j0 >> 5) - q;  // > 0: outside the band
        uint32_t hl[16];  // 8 columns of hi pairs, 8 of lo pairs
        if (off > 0) {
#pragma unroll
          for (int x = 0; x < 16; ++x) hl[x] = 0u;
        } else {
          uint32_t sreg[16];
          tmem_ld_x16(colS + j0, sreg);
          float d[16];
          const int n0 = REV ? j0 - r : r - j0;
          if (off < 0 && !edge) {
            // wholly inside the band: the powers of the nearest key's and of lambda to the 1, 2, 4 and 8, nothing to mask
            // (from a table in shared memory, which the products keep busy: a block 4000 -> 5300 clocks)
            float f[16];  // of key x, counted from the nearest
            f[0] = ex2_approx(-s2 * (float)(REV ? n0 : n0 - 15));
            f[1] = f[0] * lam1;
#pragma unroll
            for (int x = 0; x < 2; ++x) f[2 + x] = f[x] * lam2;
#pragma unroll
            for (int x = 0; x < 4; ++x) f[4 + x] = f[x] * lam4;
#pragma unroll
            for (int x = 0; x < 8; ++x) f[8 + x] = f[x] * lam8;
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 16; ++x) d[x] = __uint_as_float(sreg[x]) * f[REV ? x : 15 - x];
          } else {
            float f[16];  // (n < 0: the power is not used)
#pragma unroll
            for (int x = 0; x < 16; ++x) f[x] = ex2_approx(-s2 * (float)(REV ? n0 + x : n0 - x));
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 16; ++x) {
              const int n = REV ? n0 + x : n0 - x;
              // a select, not a multiply by zero: masked-out tokens can never leak
              d[x] = (n >= 0 && !(edge && j0 + x >= cut)) ? __uint_as_float(sreg[x]) * f[x] : 0.f;
            }
          }
#pragma unroll
          for (int x = 0; x < 8; ++x) split2(f2_pack(d[2 * x], d[2 * x + 1]), hl[x], hl[8 + x]);
        }
        tmem_st_x16(colS + j0, hl);  // in the place of the 16 fp32 columns just read
      }
      tmem_st_wait();
      tc_fence_before_sync();
      WARP_ARRIVE(V_P_READY0 + s);
    }
  } else if (warp < 20) {
    // ------------------------------------ state and fc ------------------------------------
    set_regs<V_REGS_Z, V_REGS_LAUNCH>();
    const int q = warp & 3, zh = (warp - 12) >> 2;  // features zh * 32 .. + 31 of the state, tokens zh * 64 .. + 63 of fc
    const bool lo_part = REV ? q >= 2 : q < 2;  // not the quarter that has the most scores to form
    const int e = (q & 1) * 32 + lane;          // value column
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t colDZ = lane_addr + VCOL_DZ + zh * 32, colF = lane_addr + VCOL_F + zh * 32;
    // lane l points ldmatrix at token row zh * 64 + (l >> 4) * 8 + (l & 7), value columns (q & 1) * 32 + ((l >> 3) & 1) * 8
    const uint32_t unit0 = (uint32_t)((zh * 64 + ((lane >> 4) << 3) + (lane & 7)) * 128 +
                                      ((((q & 1) * 4 + ((lane >> 3) & 1)) ^ (lane & 7)) << 4));
    float zreg[32];  // Z or Y [zh * 32 + x][e]
    auto write_state_operand = [&]() {
      unsigned char* const row = reinterpret_cast<unsigned char*>(lo_part ? sm.z[2] : sm.z[0]) + e * 128;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int at = ((zh * 4 + c) ^ (e & 7)) << 4;
        uint4 h, l;
        split2(f2_pack(zreg[c * 8 + 0], zreg[c * 8 + 1]), h.x, l.x);
        split2(f2_pack(zreg[c * 8 + 2], zreg[c * 8 + 3]), h.y, l.y);
        split2(f2_pack(zreg[c * 8 + 4], zreg[c * 8 + 5]), h.z, l.z);
        split2(f2_pack(zreg[c * 8 + 6], zreg[c * 8 + 7]), h.w, l.w);
        *reinterpret_cast<uint4*>(row + at) = h;
        if (!lo_part && split_z) *reinterpret_cast<uint4*>(row + 8192 + at) = l;
      }
      fence_proxy_async_smem();
    };
    uint32_t raw[2][16];  // c of the next block, then its fc: [16 value columns][16 tokens][8 tokens][8 value columns]
    auto fetch_c = [&](int it) {
      const uint32_t ctile = smem_u32(sm.st[it % V_STAGES].c) + unit0;
#pragma unroll
      for (int g = 0; g < 8; ++g)  // 16 tokens (g >> 1), 16 value columns (g & 1)
        ldmatrix_x4_trans((ctile ^ ((g & 1) << 5)) + (g >> 1) * 2048, raw[g & 1][(g >> 1) * 4], raw[g & 1][(g >> 1) * 4 + 1],
                          raw[g & 1][(g >> 1) * 4 + 2], raw[g & 1][(g >> 1) * 4 + 3]);
    };
    const float lam16 = ex2_approx(-s2 * 16.f);
    auto write_fc = [&](int it) {
      const int Cr = (it == (REV ? 0 : nblk - 1)) ? edge_len : 128;
      if (!lo_part || split_c) {
        float f[4];  // of this thread's token pairs in the two octets
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {  // 16 tokens, away from the edge that the state leaves through
          const int g = REV ? gi : 3 - gi;
          const int j0 = zh * 64 + g * 16 + 2 * (lane & 3);
          if (gi == 0 || Cr < 128) {
#pragma unroll
            for (int o = 0; o < 4; ++o) {
              const int j = j0 + 8 * (o >> 1) + (o & 1);
              f[o] = j < Cr ? ex2_approx(-s2 * (float)(REV ? j + 1 : Cr - 1 - j)) : 0.f;
            }
          } else {
#pragma unroll
            for (int o = 0; o < 4; ++o) f[o] *= lam16;
          }
          if (Cr < 128) {  // (what lies past the end must not come through as 0 * inf)
#pragma unroll
            for (int x = 0; x < 8; ++x) {
              const int j = j0 + 8 * ((x >> 1) & 1);
              raw[x >> 2][g * 4 + (x & 3)] &= (j < Cr ? 0xffffu : 0u) | (j + 1 < Cr ? 0xffff0000u : 0u);
            }
          }
#pragma unroll
          for (int half = 0; half < 2; ++half) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {  // octet x >> 1, value columns (x & 1) * 8
              const uint32_t w = raw[half][g * 4 + x];
              const float x0 = __uint_as_float(w << 16) * f[(x >> 1) * 2], x1 = __uint_as_float(w & 0xffff0000u) * f[(x >> 1) * 2 + 1];
              const __nv_bfloat162 hp = __floats2bfloat162_rn(x0, x1);
              uint32_t r = *reinterpret_cast<const uint32_t*>(&hp);
              if (lo_part) {
                const __nv_bfloat162 lp = __floats2bfloat162_rn(x0 - __uint_as_float(r << 16), x1 - __uint_as_float(r & 0xffff0000u));
                r = *reinterpret_cast<const uint32_t*>(&lp);
              }
              raw[half][g * 4 + x] = r;
            }
          }
        }
        // (one wide store each: a store waits its turn behind the products' accumulators, 280 clocks, whatever its width)
        tmem_st_16x128b_x8(colF, raw[0]);
        tmem_st_16x128b_x8(colF + (16u << 16), raw[1]);
        tmem_st_wait();
      }
      if (shared_tail && Cr < 128) {
        typename Sm::Stage& st = sm.st[it % V_STAGES];
        TC_WAIT_WARP_TO(fc_given_up, V_FULL_AB0 + it % V_STAGES, (it / V_STAGES) & 1, 21);
        for (int x = (warp - 12) * 32 + lane; x < (128 - Cr) * 8; x += 256) {
          reinterpret_cast<uint4*>(st.b)[Cr * 8 + x] = make_uint4(0u, 0u, 0u, 0u);
          reinterpret_cast<uint4*>(st.c)[Cr * 8 + x] = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
      }
      tc_fence_before_sync();
      WARP_ARRIVE(V_FC_READY);
      return true;
    fc_given_up:
      return false;
    };

    // the state entering the segment: see tc_walk_kernel
    {
#pragma unroll
      for (int x = 0; x < 32; ++x) zreg[x] = 0.f;
      auto add_state = [&](const float* src, bool transposed, float g) {
        if (transposed) {
          const float4* r4 = reinterpret_cast<const float4*>(src + (size_t)e * 64 + zh * 32);
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            const float4 v = ld_f4(r4 + x);
            zreg[4 * x + 0] = fmaf(g, zreg[4 * x + 0], v.x);
            zreg[4 * x + 1] = fmaf(g, zreg[4 * x + 1], v.y);
            zreg[4 * x + 2] = fmaf(g, zreg[4 * x + 2], v.z);
            zreg[4 * x + 3] = fmaf(g, zreg[4 * x + 3], v.w);
          }
        } else {
          const float* r1 = src + (size_t)(zh * 32) * 64 + e;
#pragma unroll
          for (int x = 0; x < 32; ++x) zreg[x] = fmaf(g, zreg[x], ld_f1(r1 + x * 64));
        }
      };
      if (args.follows == FOLLOWS_STATES) {
        grid_dep_wait();
        grid_dep_launch();
      }
      if (!lo_part) {
        const float reach = state_reach(s2, args.seg_len);
        const bool running = args.scanned && slow_head(s2, args.seg_len) && before > 0;
        const int near = running ? 1 : ((float)before <= reach ? before : (int)reach + 1);
        if ((near >= before || running) && job.z_in) add_state(job.z_in + (size_t)bh * 4096, job.z_in_t, 0.f);
        if (running) {
#pragma unroll
          for (int x = 0; x < 32; ++x) zreg[x] *= sm.gseg[2];
          add_state(job.local + ((size_t)bh * args.nseg + (REV ? seg + 1 : seg - 1)) * 4096, job.local_t, 1.f);
        } else {
#pragma unroll 1
          for (int k = min(near, before); k >= 1; --k) {
            const int p = REV ? seg + k : seg - k;
            add_state(job.local + ((size_t)bh * args.nseg + p) * 4096, job.local_t, sm.gseg[p == nseg_own - 1 ? 1 : 0]);
          }
        }
      }
    }
    const auto has_m3 = [&](int it) { return it + 1 < nblk || (it < nblk && last_m3); };
    if (has_m3(0)) {
      TC_WAIT_WARP(V_FULL_C0, 0, 20);
      fetch_c(0);
      if (!write_fc(0)) goto teardown;
    }
    // The value rows of the next block are fetched a block ahead, since behind the operands that the products fetch this takes 800
    // clocks (1 x 32 x 16384, bf16 results: 96 -> 92 us, dV and dK 245 -> 238) ... except where the results are twice as long and
    // use the shared memory then (fp32: 241 -> 247).
    constexpr bool AHEAD = sizeof(TOut) == 2;
    if (AHEAD && has_m3(1)) {
      TC_WAIT_WARP(V_FULL_C0 + 1, 0, 20);
      fetch_c(1);
    }
    if (has_entry) write_state_operand();
    WARP_ARRIVE(V_Z_READY);
    for (int it = 0; it < nblk; ++it) {
      const bool more = it + 1 < nblk;
      if (!more && !last_m3) break;
      const float gamma = ex2_approx(-s2 * (float)(it == (REV ? 0 : nblk - 1) ? edge_len : 128));
      if (!AHEAD && has_m3(it + 1)) {
        TC_WAIT_WARP(V_FULL_C0 + (it + 1) % V_STAGES, ((it + 1) / V_STAGES) & 1, 20);
        fetch_c(it + 1);
      }
      TC_WAIT_WARP(V_DZ_READY, it & 1, 22);
      tc_fence_after_sync();
      if (!lo_part || split_c) {
#pragma unroll
        for (int pc = 0; pc < 2; ++pc) {
          uint32_t dz[16];
          tmem_ld_x16(colDZ + pc * 16, dz);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 16; ++x) zreg[pc * 16 + x] = fmaf(gamma, zreg[pc * 16 + x], __uint_as_float(dz[x]));
        }
      }
      tc_fence_before_sync();
      if (!more) break;
      if (has_m3(it + 1) && !write_fc(it + 1)) goto teardown;
      if (AHEAD && has_m3(it + 2)) {
        TC_WAIT_WARP(V_FULL_C0 + (it + 2) % V_STAGES, ((it + 2) / V_STAGES) & 1, 20);
        fetch_c(it + 2);
      }
      TC_WAIT_WARP(V_M2_DONE, it & 1, 23);  // the state operand has been read
      write_state_operand();
      WARP_ARRIVE(V_Z_READY);
    }
    if (want_final) {
      // Z + Y, through the place of the state operand
      float* const part = reinterpret_cast<float*>(&sm.z[0][0]) + (zh * 32) * 64 + e;
      if (split_c) {
        if (lo_part) {
          TC_WAIT_WARP(V_M2_DONE, (nblk - 1) & 1, 23);
#pragma unroll
          for (int x = 0; x < 32; ++x) part[x * 64] = zreg[x];
          WARP_ARRIVE(V_FINAL);
        } else {
          TC_WAIT_WARP(V_FINAL, 0, 29);
#pragma unroll
          for (int x = 0; x < 32; ++x) zreg[x] += part[x * 64];
        }
      }
      if (!lo_part) {
        float* dst = job.final_out + (size_t)bh * 4096 + (size_t)(zh * 32) * 64 + e;
#pragma unroll
        for (int x = 0; x < 32; ++x) dst[x * 64] = zreg[x];
      }
    }
  } else {
    // ------------------------------------ output ------------------------------------
    set_regs<V_REGS_O, V_REGS_LAUNCH>();
    const int q = warp & 3, oh = (warp - 20) >> 2;  // rows q * 32 + lane, value columns oh * 32 .. + 31
    const int r = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const bool second = jobid == 0 && args.second_half && bb_ >= args.fold;  // the second half of a folded batch
    const CUtensorMap* const tm_out = second ? &maps_out.second_half : &maps_out.of[jobid];
    int staged = 0;  // blocks that left through shared memory
    for (int it = 0; it < nblk; ++it) {
      const int t0 = seg_t0 + (REV ? (nblk - 1 - it) : it) * 128;
      const int Cr = (it == (REV ? 0 : nblk - 1)) ? edge_len : 128;
      const float f = REV ? (r < Cr ? ex2_approx(-s2 * (float)(Cr - 1 - r)) : 0.f) : ex2_approx(-s2 * (float)(r + 1));
      uint32_t w[32];
      TC_WAIT_WARP(V_O_READY, it & 1, 25);
      tc_fence_after_sync();
      tmem_ld_x32(lane_addr + VCOL_OI + oh * 32, w);
      if (it > 0 || has_entry) {
#pragma unroll
        for (int pc = 0; pc < 2; ++pc) {
          uint32_t oe[16];
          tmem_ld_x16(lane_addr + VCOL_OE + oh * 32 + pc * 16, oe);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 16; ++x)
            w[pc * 16 + x] = __float_as_uint(fmaf(f, __uint_as_float(oe[x]), __uint_as_float(w[pc * 16 + x])));
        }
      } else {
        tmem_ld_wait();
      }
      tc_fence_before_sync();
      WARP_ARRIVE(V_O_FREE);
      constexpr int CHUNKS = sizeof(TOut) == 4 ? 8 : 4;  // 16 bytes each
      if (sizeof(TOut) == 2) {
#pragma unroll
        for (int x = 0; x < 16; ++x) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(w[2 * x]), __uint_as_float(w[2 * x + 1]));
          w[x] = *reinterpret_cast<const uint32_t*>(&h);
        }
      }
      if (shared_tail && Cr < 128) {
        // rows past the end are another sequence's: row by row (one block of a sequence)
        if (r < Cr) {
          uint4* dst = reinterpret_cast<uint4*>(static_cast<TOut*>(job.out) + (size_t)hh_ * args.sH + (size_t)(tok0 + t0 + r) * args.sT + oh * 32);
#pragma unroll
          for (int c = 0; c < CHUNKS; ++c) dst[c] = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
        }
        continue;
      }
      if (staged > 0) TC_WAIT_WARP(V_STORED, (staged - 1) & 1, 27);
      unsigned char* const row = sm.out[sizeof(TOut) == 4 ? oh : 0] + r * 128;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c)
        *reinterpret_cast<uint4*>(row + ((((sizeof(TOut) == 4 ? 0 : oh * 4) + c) ^ (r & 7)) << 4)) =
            make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
      fence_proxy_async_smem();
      WARP_ARRIVE(V_STAGED);
      if (warp == 20) {
        TC_WAIT_WARP(V_STAGED, staged & 1, 28);
        if (lane == 0) {
          const int batch = second ? bb_ - args.fold : bb_;
#pragma unroll
          for (int p = 0; p < (int)sizeof(TOut) / 2; ++p)  // (tokens past N are clipped by the map)
            tma_store_4d(tm_out, sm.out[p], p * 32, tok0 + t0, hh_, batch);
          tma_store_commit();
          tma_store_wait_read();
          mbar_arrive(&sm.bars[V_STORED]);
        }
        __syncwarp();
      }
      ++staged;
    }
  }

teardown:
  if (args.follows != FOLLOWS_ANY) grid_dep_wait();  // (a launch is complete only when those before it are)
  // (the bulk stores' sources were read before V_STORED; their writes complete before the kernel does)
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

template <bool REV, typename TOut>
cudaError_t launch_walk64_t(const TcMaps& m0, const TcMaps& m1, const VOutMaps& out, const TcArgs& ta, const DecayTable& tab, cudaStream_t stream) {
  const size_t smem = sizeof(VSmem<TOut>) + 1024;
  static_assert(sizeof(VSmem<TOut>) + 1024 <= 232448, "shared memory of one SM");
  auto kern = tc_walk64_kernel<REV, TOut>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  KernelTimer timer(ta.njobs == 2 ? K_WALK_PAIR : K_WALK, stream);
  err = launch_kernel(early_walks(ta.BH, ta.nseg, ta.seg_len), kern, dim3((unsigned)(ta.BH * ta.nseg * ta.njobs)), dim3(V_THREADS), smem, stream, 1, m0, m1,
                      out, ta, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}
