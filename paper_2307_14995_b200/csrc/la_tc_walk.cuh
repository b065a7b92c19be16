// Block walk for D = 128 (included by la_tc.cu, inside its anonymous namespace, after the helpers).
//
// One thread block walks the 128-token blocks of one (batch*head, segment) and produces all 128 value columns.  The
// products whose one operand is formed on chip from fp32 values are turned so that this operand is the A operand and
// lives in tensor memory (e: value columns, d: features, i, j: tokens of the block):
//   M1  S    [i, j] = a b^T                               A, B in shared memory
//   M2  O    [e, i] = Z^T a^T      Z^T  hi (+ lo)         A in tensor memory, lane e
//   M3  dZ^T [e, d] = fc^T b       fc^T hi (+ lo)         A in tensor memory, lane e     (fc = diag(f_state) c)
//   M4  O    [e, i] += c^T P^T     P    hi (+ lo)         A = c, B = P in shared memory; P is triangular, so K step k
//                                                         only runs over the columns i it reaches (N = 128 - 16 k)
// and O is scaled by diag(f_out) on the CUDA cores between M2 and M4.
// Why: a shared-memory operand pair of an M = N = 128, K = 16 instruction is 8 KB, at the 128 bytes a clock of the
// shared-memory pipe exactly the 64 clocks the instruction takes, and products win over loads: beside back-to-back
// products of that kind a dependent 4-byte load takes 130 clocks with one warp loading and 480 with sixteen (41 and 44
// without them, 64 beside products with A in tensor memory).  With [token, e] accumulators a block's products fetched
// 384 KB and the CUDA cores moved 400 KB more through the same pipe (state and fc operand tiles, the output's
// transposition); here the products fetch 290 KB, state and fc go to tensor memory, and since an accumulator lane is a
// value column, a warp's plain store instruction writes 128 contiguous bytes of one token, so that the output needs no
// transposition.
//
// Measured on B200 against a walk with [token, e] accumulators and its on-chip operands in shared memory: 7B-like shape, fp32 results, one walk
// 0.594 -> 0.467 ms, the dV and dK walks in one launch 1.186 -> 0.90 ms; 3 x 8 heads x 3001 tokens, bf16 results, one walk
// 60 -> 46 us, the pair 65 -> 50 us.
//
// Tensor memory (512 columns): R 128 (S, then dZ^T, in turn), O 128, fc^T hi/lo 2 x 64, Z^T hi/lo 2 x 64.
// Shared memory: a, b twice, c twice, P hi/lo (32 KB each).
// Order of the products per block n:  M2(n) M3(n) M4(n) M1(n+1).  They use O, R, O, R in turn, and what the CUDA cores
// do with one region happens while the next product runs in the other: S(n) is read during M2(n), O is scaled during
// M3(n), dZ(n) is read during M4(n), O(n) is stored during M1(n+1).  Shared memory is read by the CUDA cores during M2
// and M3 only (A in tensor memory), so that the value rows of the next block are fetched into registers during M3.
//
// Warp roles (28 warps): 0 TMA producer, 1 MMA issuer (all lanes converged, instructions on one elected lane), 4-19
// workers, 20-27 O group (two warps per 32 value columns, 64 tokens each).  A worker warp does, one after the other, its
// share of three jobs whose turns come at different times of a block: P (scores of up to 2 x 16 keys of 32 rows, during
// M2 and M3), Z (32 value columns x 32 features of the fp32 state in registers, from M3 on; the chain that M2 of the next
// block waits for, so it comes before F) and F (fc of 32 value columns x 32 tokens, until M3 of the next block).  With
// eight warps for P, eight for Z and four for F the state's conversion alone took 2900 of a block's 7100 clocks.
// Registers per thread after start-up: W_REGS_CTL, WRegs; they add up to what the launch has (workers with 88 and O with 64: the pair 978
// instead of 908 us at the 7B-like shape).

constexpr int W_THREADS = 896;
constexpr uint32_t WCOL_R = 0, WCOL_O = 128, WCOL_FH = 256, WCOL_FL = 320, WCOL_ZH = 384, WCOL_ZL = 448;
constexpr int W_REGS_LAUNCH = 72, W_REGS_CTL = 24;
template <int GATED>
struct WRegs {  // (the gate needs more than the plain store; with 80 for both the output group spilled: 727 -> 742 us below)
  static constexpr int W = GATED ? 72 : 96, O = GATED ? 96 : 48;
  static_assert(4 * W_REGS_CTL + 16 * W + 8 * O <= 28 * W_REGS_LAUNCH, "registers of the launch");
};

enum WBar {
  W_FULL_C0 = 0, W_FULL_C1,  // TMA -> workers, MMA: c of an even / odd block
  W_M1_OK0, W_M1_OK1,        // a and b landed (two arrivals with bytes) and the previous dZ read (16 worker warps)
  W_M2_OK,                   // state operand written (16 worker warps) and the previous O read (8 warps)
  W_M3_OK,                   // fc written and S read (16 worker warps)
  W_M4_OK,                   // P written (16 worker warps) and O scaled (8 warps)
  W_S_READY,                 // M1 done
  W_M2_DONE,                 // M2 done: O_inter complete, a and the state operand free
  // M3 done: dZ complete, b and fc free; M4 done: O complete, c and P free.  Of an even / odd block: the producer waits for
  // those of block n when nothing that M3 and M4 of block n + 1 need is still to come from it, so with one barrier they could
  // complete as well before a late producer has looked; those of block n + 2 need the loads that it starts after its wait.
  W_DZ_READY0, W_DZ_READY1,
  W_O_READY0, W_O_READY1,
  W_GATE0, W_GATE1,          // GATED: a block's sums of squares exchanged (4 warps), per half of the tokens
  W_DRAIN,
  W_NUM_BARS
};

// Arithmetic on two fp32 values in one register pair: half the issue slots, which is what the worker warps are short of
// (the reverse pair at the 1B-like shape 126 -> 123 us; in the fc conversion it spilled registers and was slower).
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// A pair as packed bf16 hi and lo terms, hi + lo = v to 2^-17.
__device__ __forceinline__ void split2(uint64_t v, uint32_t& h, uint32_t& l) {
  float a, b;
  f2_unpack(v, a, b);
  const __nv_bfloat162 hp = __floats2bfloat162_rn(a, b);
  h = *reinterpret_cast<const uint32_t*>(&hp);
  f2_unpack(f2_sub(v, f2_pack(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u))), a, b);
  const __nv_bfloat162 lp = __floats2bfloat162_rn(a, b);
  l = *reinterpret_cast<const uint32_t*>(&lp);
}

template <bool REV>
struct alignas(1024) WSmem {
  __nv_bfloat16 a[2][128 * 64];     // query-like tile, K-major, two 64-feature panels
  __nv_bfloat16 b[2][2][128 * 64];  // key-like tile, two buffers (K-major in M1, MN-major in M3)
  __nv_bfloat16 c[2][2][128 * 64];  // value-like tile, two buffers, MN-major: two 64-column chunks
  __nv_bfloat16 p_hi[2][128 * 64];  // scores, K-major: two panels of 64 keys
  __nv_bfloat16 p_lo[2][128 * 64];
  // Factor of a token's O_inter.  REV: index 1 is for the edge block (the first one walked, which may be shorter than 128
  // tokens), index 0 for every other.
  float fout[REV ? 2 : 1][128];
  float ptab[16];  // lambda^(15 - x)
  float gseg[3];   // decay through a whole segment, through the sequence's last one, and through all before this one
  uint64_t bars[W_NUM_BARS];
  uint32_t tmem_slot;
  int abort;
};

// *(p + x * stride) = v with the address as one multiply-add, which leaves the integer pipe (half rate, and what the
// conversions to hi / lo terms need) alone; one unit, so that the compiler does not hold 32 addresses in registers.
template <typename T>
__device__ __forceinline__ void store_at(T* p, uint32_t stride_bytes, int x, float v) {
  if (sizeof(T) == 4) {
    asm volatile("{\n\t.reg .b64 a;\n\tmad.wide.u32 a, %0, %1, %2;\n\tst.global.b32 [a], %3;\n\t}" ::"r"(stride_bytes),
                 "r"((uint32_t)x), "l"(reinterpret_cast<uint64_t>(p)), "f"(v)
                 : "memory");
  } else {
    asm volatile("{\n\t.reg .b64 a;\n\tmad.wide.u32 a, %0, %1, %2;\n\tst.global.b16 [a], %3;\n\t}" ::"r"(stride_bytes),
                 "r"((uint32_t)x), "l"(reinterpret_cast<uint64_t>(p)), "h"(__bfloat16_as_ushort(__float2bfloat16_rn(v)))
                 : "memory");
  }
}

// The same if x < end, without a branch.
template <typename T>
__device__ __forceinline__ void store_below(T* p, uint32_t stride_bytes, int x, float v, int end) {
  if (sizeof(T) == 4) {
    asm volatile(
        "{\n\t.reg .b64 a;\n\t.reg .pred in;\n\tsetp.gt.s32 in, %4, %1;\n\tmad.wide.u32 a, %0, %1, %2;\n\t"
        "@in st.global.b32 [a], %3;\n\t}" ::"r"(stride_bytes),
        "r"((uint32_t)x), "l"(reinterpret_cast<uint64_t>(p)), "f"(v), "r"(end)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .b64 a;\n\t.reg .pred in;\n\tsetp.gt.s32 in, %4, %1;\n\tmad.wide.u32 a, %0, %1, %2;\n\t"
        "@in st.global.b16 [a], %3;\n\t}" ::"r"(stride_bytes),
        "r"((uint32_t)x), "l"(reinterpret_cast<uint64_t>(p)), "h"(__bfloat16_as_ushort(__float2bfloat16_rn(v))), "r"(end)
        : "memory");
  }
}

// The 32 bits at p + x * stride, likewise.
__device__ __forceinline__ uint32_t load_u32_at(const void* p, uint32_t stride_bytes, int x) {
  uint32_t r;
  asm volatile("{\n\t.reg .b64 a;\n\tmad.wide.u32 a, %1, %2, %3;\n\tld.global.b32 %0, [a];\n\t}"
               : "=r"(r)
               : "r"(stride_bytes), "r"((uint32_t)x), "l"(reinterpret_cast<uint64_t>(p)));
  return r;
}

// Sum over the eight lanes with the same lane % 4 of each of 16 values per lane; the lane returns the totals of values
// 2 (lane / 4) and 2 (lane / 4) + 1.
__device__ __forceinline__ float2 octet_sums(const float (&v)[16], int lane) {
  float t[8], r[4];
  const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0, b2 = (lane & 4) != 0;
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const float keep = b4 ? v[8 + x] : v[x], send = b4 ? v[x] : v[8 + x];
    t[x] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const float keep = b3 ? t[4 + x] : t[x], send = b3 ? t[x] : t[4 + x];
    r[x] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  const float k0 = b2 ? r[2] : r[0], s0 = b2 ? r[0] : r[2], k1 = b2 ? r[3] : r[1], s1 = b2 ? r[1] : r[3];
  return make_float2(k0 + __shfl_xor_sync(0xffffffffu, s0, 4), k1 + __shfl_xor_sync(0xffffffffu, s1, 4));
}

// args.njobs == 2: two walks of the same direction over the same tokens in one launch (the dV and dK walks of the
// backward pass, which between them read Q, K, V and dO); the thread blocks of the two jobs alternate, so that the two
// readers of a tile run side by side and the tile comes from HBM once.
// GATED (forward, single job): the epilogue y = SRMSNorm(out) (.) u of Eq. 3 with Eq. 8 is applied to the rows
// before they leave (job.u, job.y; job.rstd optional); 1: y alone, 2: out as well.
// EARLY: launched while the launch before it ends (see Follows).
template <bool REV, typename TOut, int GATED, bool EARLY>
__global__ void __launch_bounds__(W_THREADS, 1)
tc_walk_kernel(const __grid_constant__ TcMaps maps0, const __grid_constant__ TcMaps maps1,
               const __grid_constant__ TcArgs args, const __grid_constant__ DecayTable tab) {
  extern __shared__ unsigned char smem_raw[];
  WSmem<REV>& sm = *reinterpret_cast<WSmem<REV>*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (EARLY && args.follows == FOLLOWS_ANY && args.seq_start) grid_dep_wait();  // the tables of a packed batch
  const int jobid = (args.njobs == 2) ? (int)(blockIdx.x & 1) : 0;
  const int bidx = (args.njobs == 2) ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const TcJob& job = args.job[jobid];
  const int seg = bidx % args.nseg;
  int bh = bidx / args.nseg;
  // packed batch: thread blocks take the sequences longest first, so that a long one is not what the launch ends on
  if (args.seq_order) bh = args.seq_order[bh / args.H] * args.H + bh % args.H;
  // Packed batch: "batch" entry bh / H is a sequence of its own length inside one [tokens, H, D] tensor; tok0 is its
  // first token, and the maps' batch coordinate is 0.  Dense batch: tok0 = 0, every entry has N tokens.
  const int n_tok = args.seq_len ? args.seq_len[bh / args.H] : args.N;
  const int tok0 = args.seq_start ? args.seq_start[bh / args.H] : 0;
  const int nseg_own = (n_tok + args.seg_len - 1) / args.seg_len;
  if (seg >= nseg_own) return;  // the grid covers the longest sequence; nothing has been set up yet
  const int seg_t0 = seg * args.seg_len;
  const int seg_t1 = min(n_tok, seg_t0 + args.seg_len);
  const int nblk = (seg_t1 - seg_t0 + 127) >> 7;
  const int edge_len = seg_t1 - seg_t0 - (nblk - 1) * 128;  // tokens of the block that holds the segment's last ones
  const float s2 = (float)tab.s2[bh % args.H];
  const int before = REV ? nseg_own - 1 - seg : seg;  // segments walked before this one
  const bool has_entry = job.z_in != nullptr || before > 0;  // else the first block has no O_inter: M2 is skipped
  const bool want_final = job.final_out && (REV ? seg == 0 : seg == nseg_own - 1);

  if (tid == 0) {
    for (int i = 0; i < W_NUM_BARS; ++i) {
      uint32_t count = 1;
      if (i == W_M1_OK0 || i == W_M1_OK1) count = 18;
      if (i == W_M2_OK || i == W_M4_OK) count = 24;
      if (i == W_M3_OK) count = 16;
      if (i == W_GATE0 || i == W_GATE1) count = 4;
      mbar_init(&sm.bars[i], count);
    }
    sm.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    if (EARLY && args.follows == FOLLOWS_ANY) grid_dep_wait();  // (see Follows)
    tmem_alloc(&sm.tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  if (warp >= 4 && warp < 12) {
    const int x = tid - 128, set = x >> 7, i = x & 127;
    if (REV) {
      const int Cr = set ? edge_len : 128;
      sm.fout[REV ? set : 0][i] = i < Cr ? ex2_approx(-s2 * (float)(Cr - 1 - i)) : 0.f;
    } else if (set == 0) {
      sm.fout[0][i] = ex2_approx(-s2 * (float)(i + 1));
    }
    if (x >= 192 && x < 195) {
      const int len = x == 192 ? args.seg_len : x == 193 ? n_tok - (nseg_own - 1) * args.seg_len : REV ? n_tok - seg_t1 : seg_t0;
      sm.gseg[x - 192] = decay_pow_d(tab.s2[bh % args.H], (double)len);
    }
    if (x < 16) sm.ptab[x] = ex2_approx(-s2 * (float)(15 - x));
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sm.tmem_slot;
  if (EARLY && args.follows == FOLLOWS_ANY) {
    grid_dep_wait();
    grid_dep_launch();
  }
  if (warp < 4) {
    set_regs<W_REGS_CTL, W_REGS_LAUNCH>();
    if (warp == 0) {
      // ------------------------------------ TMA producer ------------------------------------
      if (lane == 0) {
        int armed_ab = 0, armed_c = 0;  // blocks whose loads have been started
        const TcMaps* const maps = jobid ? &maps1 : &maps0;
        const int hh_ = bh % args.H;  // head coordinate of the 4-D tensor maps
        const int bb_ = args.seq_start ? 0 : bh / args.H;
        const int bf_ = args.fold && bb_ >= args.fold ? bb_ - args.fold : bb_;  // of an operand that is shared
        auto token = [&](int it) { return tok0 + seg_t0 + (REV ? (nblk - 1 - it) : it) * 128; };
        auto load = [&](int bar_id, __nv_bfloat16* dst, const CUtensorMap* map, int it, int batch) {
          uint64_t* bar = &sm.bars[bar_id];
          mbar_arrive_expect_tx(bar, 32768);
          tma_load_4d(dst, map, bar, 0, token(it), hh_, batch);
          tma_load_4d(dst + 128 * 64, map, bar, 64, token(it), hh_, batch);
        };
        const int ba = job.shared & SHARED_A ? bf_ : bb_, bb = job.shared & SHARED_B ? bf_ : bb_, bc = job.shared & SHARED_C ? bf_ : bb_;
        auto load_a = [&](int it) { load(W_M1_OK0 + (it & 1), &sm.a[0][0], &maps->a, it, ba); };
        auto load_b = [&](int it) { load(W_M1_OK0 + (it & 1), &sm.b[it & 1][0][0], &maps->b, it, bb); armed_ab = it + 1; };
        auto load_c = [&](int it) { load(W_FULL_C0 + (it & 1), &sm.c[it & 1][0][0], &maps->c, it, bc); armed_c = it + 1; };
        load_b(0);
        load_a(0);
        load_c(0);
        if (nblk > 1) {
          load_b(1);
          load_c(1);
        }
        for (int it = 0; it + 1 < nblk; ++it) {
          TC_WAIT_TO(producer_done, W_M2_DONE, it & 1, 3);
          load_a(it + 1);
          if (it + 2 < nblk) {
            TC_WAIT_TO(producer_done, W_DZ_READY0 + (it & 1), (it >> 1) & 1, 5);
            load_b(it + 2);
            TC_WAIT_TO(producer_done, W_O_READY0 + (it & 1), (it >> 1) & 1, 2);
            load_c(it + 2);
          }
        }
      producer_done:
        // After an expired wait: nothing may be in flight when the block exits.  (A block that gave up before the Z group's
        // arrivals leaves the a / b phases incomplete; these waits are bounded like every other.)
        if (sm.abort) {
          for (int k = 0; k < 2; ++k) {
            const int ab = armed_ab - 1 - k, cc = armed_c - 1 - k;
            if (ab >= 0) drain_wait(&sm.bars[W_M1_OK0 + (ab & 1)], (ab >> 1) & 1);
            if (cc >= 0) drain_wait(&sm.bars[W_FULL_C0 + (cc & 1)], (cc >> 1) & 1);
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------ MMA issuer ------------------------------------
      constexpr uint32_t ID_KK = umma_idesc_bf16(128, 128, false, false);  // K-major or tensor-memory A x K-major B
      constexpr uint32_t ID_KN = umma_idesc_bf16(128, 128, false, true);   // tensor-memory A x MN-major B
      constexpr uint32_t HI = UMMA_DESC_HI_SBO1024;
      const uint32_t go = elect_one();
      const bool split_p = (args.precision & 1) != 0, split_z = (args.precision & 2) != 0;
      const bool split_c = (args.precision & 4) != 0 && s2 != 0.f;  // lambda == 1: the lo term is identically zero
      // Low descriptor halves as one run-time base plus constants (16-byte units): this warp's few registers must hold
      // everything, since a spilled value comes back through the pipe that the products keep busy.
      using Sm = WSmem<REV>;
      const uint32_t base = (smem_u32(&sm) & 0x3FFFFu) >> 4;
      constexpr uint32_t KMAJ = 1u << 16, MNMAJ = 1024u << 16;  // leading-dimension offset 16 bytes / 16 KB
      constexpr uint32_t OA = (uint32_t)(offsetof(Sm, a) >> 4) + KMAJ, OB = (uint32_t)(offsetof(Sm, b) >> 4);
      constexpr uint32_t OC = (uint32_t)(offsetof(Sm, c) >> 4) + MNMAJ;
      constexpr uint32_t OPH = (uint32_t)(offsetof(Sm, p_hi) >> 4) + KMAJ, OPL = (uint32_t)(offsetof(Sm, p_lo) >> 4) + KMAJ;
      TC_WAIT_WARP_TO(mma_done, W_M1_OK0, 0, 7);
      tc_fence_after_sync();
      umma_group_ss<8, true, true>(tmem + WCOL_R, base + OA, base + OB + KMAJ, HI, ID_KK, 0, go);
      umma_commit_if(&sm.bars[W_S_READY], go);
      for (int it = 0; it < nblk; ++it) {
        const uint32_t par = it & 1;
        const bool inter = it > 0 || has_entry;
        const uint32_t buf = base + par * 2048;  // base of this block's b and c buffers
        TC_WAIT_WARP_TO(mma_done, W_M2_OK, par, 12);
        tc_fence_after_sync();
        if (inter) {
          umma_group_tsd<true>(tmem + WCOL_O, tmem + WCOL_ZH, base + OA, HI, ID_KK, 0, go);
          if (split_z) umma_group_tsd<true>(tmem + WCOL_O, tmem + WCOL_ZL, base + OA, HI, ID_KK, 1, go);
        }
        umma_commit_if(&sm.bars[W_M2_DONE], go);
        if (it + 1 < nblk || want_final) {  // the state after the segment's last block is often not wanted
          TC_WAIT_WARP_TO(mma_done, W_M3_OK, par, 13);
          tc_fence_after_sync();
          umma_group_tsd<false>(tmem + WCOL_R, tmem + WCOL_FH, buf + OB + MNMAJ, HI, ID_KN, 0, go);
          if (split_c) umma_group_tsd<false>(tmem + WCOL_R, tmem + WCOL_FL, buf + OB + MNMAJ, HI, ID_KN, 1, go);
        }
        umma_commit_if(&sm.bars[W_DZ_READY0 + par], go);
        TC_WAIT_WARP_TO(mma_done, W_FULL_C0 + par, (it >> 1) & 1, 15);
        TC_WAIT_WARP_TO(mma_done, W_M4_OK, par, 14);
        tc_fence_after_sync();
        umma_tri4<REV ? 7 : 0, REV>(tmem + WCOL_O, buf + OC, base + OPH, HI, inter ? 1u : 0u, go);
        umma_tri4<REV ? 3 : 4, REV>(tmem + WCOL_O, buf + OC, base + OPH, HI, 1, go);
        if (split_p) {
          umma_tri4<REV ? 7 : 0, REV>(tmem + WCOL_O, buf + OC, base + OPL, HI, 1, go);
          umma_tri4<REV ? 3 : 4, REV>(tmem + WCOL_O, buf + OC, base + OPL, HI, 1, go);
        }
        umma_commit_if(&sm.bars[W_O_READY0 + par], go);
        if (it + 1 < nblk) {
          TC_WAIT_WARP_TO(mma_done, W_M1_OK0 + (par ^ 1), ((it + 1) >> 1) & 1, 11);
          tc_fence_after_sync();
          umma_group_ss<8, true, true>(tmem + WCOL_R, base + OA, base + (par ^ 1) * 2048 + OB + KMAJ, HI, ID_KK, 0, go);
          umma_commit_if(&sm.bars[W_S_READY], go);
        }
      }
    mma_done:
      if (sm.abort) {
        umma_commit_if(&sm.bars[W_DRAIN], go);
        drain_wait(&sm.bars[W_DRAIN], 0);
      }
    }
  } else if (warp < 20) {
    // ------------------------------------ workers ------------------------------------
    set_regs<WRegs<GATED>::W, W_REGS_LAUNCH>();
    const int q = warp & 3;                // quarter of tensor memory: score rows / value columns q * 32 + lane
    const int w4 = (warp - 4) >> 2;        // this warp's share within the quarter
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t colDZ = lane_addr + WCOL_R + w4 * 32;
    const uint32_t colZ = lane_addr + WCOL_ZH + w4 * 16;  // (the lo terms follow 64 columns further)
    const uint32_t colF = lane_addr + WCOL_FH + w4 * 16;
    const bool split_p = (args.precision & 1) != 0, split_z = (args.precision & 2) != 0;
    const bool split_c = (args.precision & 4) != 0 && s2 != 0.f;
    // P: the 16-key pieces w4 and w4 + 4 of the band's 2 (q + 1), forward from key 0, reverse from key 127 downwards
    const int pieces = (REV ? 4 - q : q + 1) * 2;
    const int n_pieces = w4 < pieces ? (w4 + 4 < pieces ? 2 : 1) : 0;
    // Reverse walk of a packed batch: the keys past the end of the sequence lie inside the band of the edge block, and
    // there they are the next sequence's tokens, not the zero fill a dense batch has.
    const int cut = (REV && args.seq_start) ? edge_len : 128;
    // F: lane l points ldmatrix at token row w4 * 32 + (l >> 4) * 8 + (l & 7), value columns q * 32 + ((l >> 3) & 1) * 8
    const uint32_t unit0 = (uint32_t)((q >> 1) * 16384 + (w4 * 32 + ((lane >> 4) << 3) + (lane & 7)) * 128 +
                                      ((((q & 1) * 4 + ((lane >> 3) & 1)) ^ (lane & 7)) << 4));
    const bool need_state = nblk > 1 || want_final;

    float zreg[32];    // Z[w4 * 32 + x][value column q * 32 + lane]
    uint32_t raw[16];  // c of the next block: [16 tokens][16 value columns][8 tokens][8 value columns]
    auto write_state_operand = [&]() {
#pragma unroll
      for (int pc = 0; pc < 4; ++pc) {
        uint4 h, l;
        split2(f2_pack(zreg[pc * 8 + 0], zreg[pc * 8 + 1]), h.x, l.x);
        split2(f2_pack(zreg[pc * 8 + 2], zreg[pc * 8 + 3]), h.y, l.y);
        split2(f2_pack(zreg[pc * 8 + 4], zreg[pc * 8 + 5]), h.z, l.z);
        split2(f2_pack(zreg[pc * 8 + 6], zreg[pc * 8 + 7]), h.w, l.w);
        tmem_st_x4(colZ + pc * 4, h);
        if (split_z) tmem_st_x4(colZ + 64 + pc * 4, l);
      }
      tmem_st_wait();
      tc_fence_before_sync();
    };
    auto fetch_c = [&](int it) {
      const uint32_t ctile = smem_u32(&sm.c[it & 1][0][0]) + unit0;
#pragma unroll
      for (int g = 0; g < 4; ++g)  // 16 tokens (g >> 1), 16 value columns (g & 1)
        ldmatrix_x4_trans((ctile ^ ((g & 1) << 5)) + (g >> 1) * 2048, raw[4 * g], raw[4 * g + 1], raw[4 * g + 2], raw[4 * g + 3]);
    };
    // fc^T = (diag(f_state) c)^T: ldmatrix has transposed 8 x 8 pieces of the c tile, a register holds a token pair of one
    // value column, as the A operand wants it
    auto write_fc = [&](int it) {
      const int Cr = (it == (REV ? 0 : nblk - 1)) ? edge_len : 128;
#pragma unroll
      for (int g2 = 0; g2 < 2; ++g2) {  // 16 tokens
        float f[4];                     // of this thread's token pairs in the two octets
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int j = w4 * 32 + g2 * 16 + 8 * (o >> 1) + 2 * (lane & 3) + (o & 1);
          f[o] = j < Cr ? ex2_approx(-s2 * (float)(REV ? j + 1 : Cr - 1 - j)) : 0.f;
        }
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t h[4], l[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {  // octet x >> 1, value columns (x & 1) * 8
            const uint32_t w = raw[g2 * 8 + half * 4 + x];
            const float x0 = __uint_as_float(w << 16) * f[(x >> 1) * 2], x1 = __uint_as_float(w & 0xffff0000u) * f[(x >> 1) * 2 + 1];
            const __nv_bfloat162 hp = __floats2bfloat162_rn(x0, x1);
            h[x] = *reinterpret_cast<const uint32_t*>(&hp);
            const __nv_bfloat162 lp =
                __floats2bfloat162_rn(x0 - __uint_as_float(h[x] << 16), x1 - __uint_as_float(h[x] & 0xffff0000u));
            l[x] = *reinterpret_cast<const uint32_t*>(&lp);
          }
          const uint32_t at = colF + ((uint32_t)(half * 16) << 16) + g2 * 8;
          tmem_st_16x128b_x2(at, h);
          if (split_c) tmem_st_16x128b_x2(at + 64, l);
        }
      }
      tmem_st_wait();
      tc_fence_before_sync();
    };

    // The state entering the segment: z = z_in, then z <- lambda^(length) z + local state for the segments before this one.
    // Only the nearest `near` of them are read: through so many whole segments the decay is below 2^-160, exactly zero in
    // fp32.  Where a launch has made running sums of the slow heads' states (args.scanned), one state and z_in are enough.
    // (A head that decays reads one state; a slow one all of them, about 1 us each, against 5 us for the extra launch.)
    {
      // (written so that the compiler does not know the zeros: with them it spilled the copies it made of this part)
#pragma unroll
      for (int x = 0; x < 32; ++x) asm volatile("mov.b32 %0, 0;" : "=f"(zreg[x]));
      auto add_state = [&](const float* src, bool transposed, float g) {
        if (transposed) {
          const float4* r4 = reinterpret_cast<const float4*>(src + (size_t)(q * 32 + lane) * 128 + w4 * 32);
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            const float4 v = ld_f4(r4 + x);
            zreg[4 * x + 0] = fmaf(g, zreg[4 * x + 0], v.x);
            zreg[4 * x + 1] = fmaf(g, zreg[4 * x + 1], v.y);
            zreg[4 * x + 2] = fmaf(g, zreg[4 * x + 2], v.z);
            zreg[4 * x + 3] = fmaf(g, zreg[4 * x + 3], v.w);
          }
        } else {
          const float* r1 = src + (size_t)(w4 * 32) * 128 + q * 32 + lane;
#pragma unroll
          for (int x = 0; x < 32; ++x) zreg[x] = fmaf(g, zreg[x], ld_f1(r1 + x * 128));
        }
      };
      if (EARLY && args.follows == FOLLOWS_STATES) {
        grid_dep_wait();
        grid_dep_launch();
      }
      const float reach = state_reach(s2, args.seg_len);
      const bool running = args.scanned && slow_head(s2, args.seg_len) && before > 0;
      const int near = running ? 1 : ((float)before <= reach ? before : (int)reach + 1);
      if ((near >= before || running) && job.z_in) add_state(job.z_in + (size_t)bh * (128 * 128), job.z_in_t, 0.f);
      if (running) {
#pragma unroll
        for (int x = 0; x < 32; ++x) zreg[x] *= sm.gseg[2];
        add_state(job.local + ((size_t)bh * args.nseg + (REV ? seg + 1 : seg - 1)) * (128 * 128), job.local_t, 1.f);
      } else {
#pragma unroll 1
        for (int k = min(near, before); k >= 1; --k) {
          const int p = REV ? seg + k : seg - k;
          if (k >= 2 && !job.local_t) {  // two states' loads in flight
            const float g1 = sm.gseg[p == nseg_own - 1 ? 1 : 0], g2 = sm.gseg[0];
            const float* r1 = job.local + ((size_t)bh * args.nseg + p) * (128 * 128) + (size_t)(w4 * 32) * 128 + q * 32 + lane;
            const float* r2 = r1 + (REV ? -1 : 1) * (128 * 128);
            float v[32];
#pragma unroll
            for (int x = 0; x < 32; ++x) v[x] = ld_f1(r1 + x * 128);
#pragma unroll
            for (int x = 0; x < 32; ++x) zreg[x] = fmaf(g2, fmaf(g1, zreg[x], v[x]), ld_f1(r2 + x * 128));
            --k;
            continue;
          }
          add_state(job.local + ((size_t)bh * args.nseg + p) * (128 * 128), job.local_t, sm.gseg[p == nseg_own - 1 ? 1 : 0]);
        }
      }
    }
    WARP_ARRIVE(W_M1_OK0);  // there is no earlier dZ to read
    if (has_entry) write_state_operand();
    WARP_ARRIVE(W_M2_OK);
    if (need_state) {
      TC_WAIT_WARP(W_FULL_C0, 0, 20);
      fetch_c(0);
      write_fc(0);
    }
    for (int it = 0; it < nblk; ++it) {
      // ---- P: S -> masked, decayed bf16 hi / lo rows in shared memory (what lies outside the band is never read) ----
      TC_WAIT_WARP(W_S_READY, it & 1, 17);
      tc_fence_after_sync();
      if (n_pieces == 0) WARP_ARRIVE(W_M3_OK);
#pragma unroll 1
      for (int pi = 0; pi < n_pieces; ++pi) {
        const int r = q * 32 + lane;  // score row
        const int j0 = REV ? 112 - 16 * (w4 + 4 * pi) : 16 * (w4 + 4 * pi);
        uint32_t sreg[16];
        tmem_ld_x16(lane_addr + WCOL_R + j0, sreg);
        const bool edge = REV && it == 0 && cut < 128;
        const float base = ex2_approx(-s2 * (float)(REV ? j0 - r : r - j0 - 15));
        tmem_ld_wait();
        if (pi == n_pieces - 1) {
          tc_fence_before_sync();
          WARP_ARRIVE(W_M3_OK);  // all of S that this warp needs is in registers, and its fc is written
        }
        float d[16];
        if ((j0 >> 5) != q && !edge) {
          // wholly inside the band: lambda^|i-j| = row factor * table entry (both at most 1), nothing to mask
#pragma unroll
          for (int x4 = 0; x4 < 4; ++x4) {
            const float4 t = *reinterpret_cast<const float4*>(&sm.ptab[REV ? 12 - 4 * x4 : 4 * x4]);
            d[4 * x4 + 0] = __uint_as_float(sreg[4 * x4 + 0]) * base * (REV ? t.w : t.x);
            d[4 * x4 + 1] = __uint_as_float(sreg[4 * x4 + 1]) * base * (REV ? t.z : t.y);
            d[4 * x4 + 2] = __uint_as_float(sreg[4 * x4 + 2]) * base * (REV ? t.y : t.z);
            d[4 * x4 + 3] = __uint_as_float(sreg[4 * x4 + 3]) * base * (REV ? t.x : t.w);
          }
        } else {
          const int n0 = REV ? j0 - r : r - j0;
#pragma unroll
          for (int x = 0; x < 16; ++x) {
            const int n = REV ? n0 + x : n0 - x;
            // a select, not a multiply by zero: masked-out tokens can never leak (n < 0: the power is not used)
            const float f = ex2_approx(-s2 * (float)n);
            d[x] = (n >= 0 && !(edge && j0 + x >= cut)) ? __uint_as_float(sreg[x]) * f : 0.f;
          }
        }
        uint32_t h8[8], l8[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) split2(f2_pack(d[2 * x], d[2 * x + 1]), h8[x], l8[x]);
        unsigned char* const row = reinterpret_cast<unsigned char*>(&sm.p_hi[j0 >> 6][0]) + r * 128;
        const int u0 = ((((j0 & 63) >> 3)) ^ (r & 7)) << 4, u1 = u0 ^ 16;
        *reinterpret_cast<uint4*>(row + u0) = make_uint4(h8[0], h8[1], h8[2], h8[3]);
        *reinterpret_cast<uint4*>(row + u1) = make_uint4(h8[4], h8[5], h8[6], h8[7]);
        if (split_p) {
          *reinterpret_cast<uint4*>(row + sizeof(sm.p_hi) + u0) = make_uint4(l8[0], l8[1], l8[2], l8[3]);
          *reinterpret_cast<uint4*>(row + sizeof(sm.p_hi) + u1) = make_uint4(l8[4], l8[5], l8[6], l8[7]);
        }
      }
      fence_proxy_async_smem();
      WARP_ARRIVE(W_M4_OK);
      const bool more = it + 1 < nblk;
      if (!more && !want_final) break;
      if (more) {
        TC_WAIT_WARP(W_FULL_C0 + ((it + 1) & 1), ((it + 1) >> 1) & 1, 20);
        fetch_c(it + 1);
      }
      // ---- Z <- Gamma Z + dZ ----
      const float gamma = ex2_approx(-s2 * (float)(it == (REV ? 0 : nblk - 1) ? edge_len : 128));
      TC_WAIT_WARP(W_DZ_READY0 + (it & 1), (it >> 1) & 1, 22);  // M2 and M3 of this block are done
      tc_fence_after_sync();
#pragma unroll
      for (int pc = 0; pc < 2; ++pc) {
        uint32_t dh[16];
        tmem_ld_x16(colDZ + pc * 16, dh);
        tmem_ld_wait();
#pragma unroll
        for (int x = 0; x < 16; x += 2)
          f2_unpack(f2_fma(f2_pack(gamma, gamma), f2_pack(zreg[pc * 16 + x], zreg[pc * 16 + x + 1]),
                           f2_pack(__uint_as_float(dh[x]), __uint_as_float(dh[x + 1]))),
                    zreg[pc * 16 + x], zreg[pc * 16 + x + 1]);
      }
      tc_fence_before_sync();
      if (more) {
        WARP_ARRIVE(W_M1_OK0 + ((it + 1) & 1));  // M1 of the next block may overwrite dZ
        write_state_operand();
        WARP_ARRIVE(W_M2_OK);
        write_fc(it + 1);
      }
    }
    if (want_final) {
      float* dst = job.final_out + (size_t)bh * (128 * 128) + (size_t)(w4 * 32) * 128 + q * 32 + lane;
#pragma unroll
      for (int x = 0; x < 32; ++x) dst[x * 128] = zreg[x];
    }
  } else {
    // ------------------------------------ O group ------------------------------------
    set_regs<WRegs<GATED>::O, W_REGS_LAUNCH>();
    const int q = warp & 3;
    const int th = (warp >= 24) ? 64 : 0;  // first of this warp's 64 tokens
    const uint32_t colO = tmem + ((uint32_t)(q * 32) << 16) + WCOL_O + th;
    const int batch = args.seq_start ? 0 : bh / args.H;
    const size_t head_off = (size_t)batch * args.sB + (size_t)(bh % args.H) * args.sH + (size_t)tok0 * args.sT;
    // (one addition, 0 where there is no second tensor: a second pointer in the job made the 3 x 8 heads x 3001 step 1 % slower)
    TOut* const out = reinterpret_cast<TOut*>(static_cast<char*>(job.out) + (jobid == 0 && batch >= args.fold ? args.second_half : 0)) +
                      head_off + q * 32 + lane;
    WARP_ARRIVE(W_M2_OK);  // there is no earlier O to read
    for (int it = 0; it < nblk; ++it) {
      // ---- O <- O diag(f_out), between M2 and M4 ----
      TC_WAIT_WARP(W_M2_DONE, it & 1, 24);
      if (it > 0 || has_entry) {
        const float* const ft = &sm.fout[REV && it == 0 ? 1 : 0][th];
        tc_fence_after_sync();
#pragma unroll 1
        for (int pc = 0; pc < 4; ++pc) {
          uint32_t w[16];
          tmem_ld_x16(colO + pc * 16, w);
          tmem_ld_wait();
#pragma unroll
          for (int x4 = 0; x4 < 4; ++x4) {
            const float4 t = *reinterpret_cast<const float4*>(ft + pc * 16 + 4 * x4);
            w[4 * x4 + 0] = __float_as_uint(__uint_as_float(w[4 * x4 + 0]) * t.x);
            w[4 * x4 + 1] = __float_as_uint(__uint_as_float(w[4 * x4 + 1]) * t.y);
            w[4 * x4 + 2] = __float_as_uint(__uint_as_float(w[4 * x4 + 2]) * t.z);
            w[4 * x4 + 3] = __float_as_uint(__uint_as_float(w[4 * x4 + 3]) * t.w);
          }
          tmem_st_x16(colO + pc * 16, w);
        }
        tmem_st_wait();
        tc_fence_before_sync();
      }
      WARP_ARRIVE(W_M4_OK);
      // ---- store O ----
      const int t0 = seg_t0 + (REV ? (nblk - 1 - it) : it) * 128 + th;
      const int rows = seg_t1 - t0;  // tokens of this warp's 64 that exist (may be <= 0)
      TOut* dst = out + (size_t)t0 * args.sT;
      // u of this warp's 64 tokens, two value columns to a register: lanes 0..15 hold token 2 x, lanes 16..31 token 2 x + 1
      uint32_t upair[GATED ? 32 : 1];
      if constexpr (GATED != 0) {
        const __nv_bfloat16* up = static_cast<const __nv_bfloat16*>(job.u) + head_off +
                                  (size_t)(t0 + (lane >> 4)) * args.sT + q * 32 + (lane & 15) * 2;
        const int mine = rows - (lane >> 4);
#pragma unroll
        for (int x = 0; x < 32; ++x) {
          upair[x] = 0u;
          if (2 * x < mine) upair[x] = load_u32_at(up, (uint32_t)args.sT * 4u, x);
        }
      }
      TC_WAIT_WARP(W_O_READY0 + (it & 1), (it >> 1) & 1, 25);
      tc_fence_after_sync();
      const uint32_t stride = (uint32_t)args.sT * (uint32_t)sizeof(TOut);
      if constexpr (GATED != 0) {
        // Sums of squares of 64 tokens over this quarter's value columns (lanes), exchanged between the four quarters through
        // shared memory.  They are read in the 16 x 256-bit shape, which has four lanes of a token in one thread, so that 14
        // shuffles add up what 64 would.  The factors come back by a broadcast read, O in pieces of 16 tokens, two of them
        // ahead, so that M2 of the next block may overwrite it when half is stored, and a token past the end costs a
        // predicate instead of a branch, which kept the loads and shuffles of different tokens from overlapping.
        // 7B-like shape, la_fwd_gated: y alone 983 -> 727 us in fp32, 952 -> 695 in bf16; with o 978 (o to memory, then a row
        // kernel) -> 837 and 987 -> 771; 2 x 16 x 8192 in fp32 145 -> 110, with o 138 -> 129.
        // (The buffers are a part of the score tile that the forward walk never uses: keys 64.. of rows 0..15 for the sums and
        // of rows 16..31 for the factors.  A warp has read a block's sums before it arrives for M4 of the next block, which
        // the others' next sums wait for.)
        float(*const g)[64] = reinterpret_cast<float(*)[64]>(&sm.p_hi[1][0]) + (th >> 6) * 4;
        float* const factor = reinterpret_cast<float*>(&sm.p_hi[1][16 * 64]) + (warp - 20) * 64;
        {
          float s[16];  // tokens 8 i + 2 (lane % 4) + c at 2 i + c
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            uint32_t w[32];
            tmem_ld_16x256b_x8(colO + ((uint32_t)(half * 16) << 16), w);
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 16; ++x) {
              const float v0 = __uint_as_float(w[(x >> 1) * 4 + (x & 1)]), v1 = __uint_as_float(w[(x >> 1) * 4 + 2 + (x & 1)]);
              s[x] = half ? fmaf(v0, v0, fmaf(v1, v1, s[x])) : fmaf(v0, v0, v1 * v1);
            }
          }
          *reinterpret_cast<float2*>(&g[q][2 * lane]) = octet_sums(s, lane);
        }
        WARP_ARRIVE(W_GATE0 + (th >> 6));
        uint32_t o[32];
        tmem_ld_x32(colO, o);
        TC_WAIT_WARP(W_GATE0 + (th >> 6), it & 1, 26);
        {
          float2 f;  // of tokens 2 lane, 2 lane + 1
          const float2 a = *reinterpret_cast<const float2*>(&g[0][2 * lane]), b = *reinterpret_cast<const float2*>(&g[1][2 * lane]);
          const float2 c = *reinterpret_cast<const float2*>(&g[2][2 * lane]), d = *reinterpret_cast<const float2*>(&g[3][2 * lane]);
          f.x = (a.x + b.x) + (c.x + d.x);
          f.y = (a.y + b.y) + (c.y + d.y);
          f.x = f.x > 0.f ? rsqrtf(f.x * (1.f / 128.f)) : 0.f;
          f.y = f.y > 0.f ? rsqrtf(f.y * (1.f / 128.f)) : 0.f;
          *reinterpret_cast<float2*>(&factor[2 * lane]) = f;
          if (job.rstd && q == 0) {  // rstd has the layout of the token tensors without the feature dimension
            const size_t at = (head_off + (size_t)(t0 + 2 * lane) * args.sT) >> 7;
            if (2 * lane < rows) job.rstd[at] = f.x;
            if (2 * lane + 1 < rows) job.rstd[at + (args.sT >> 7)] = f.y;
          }
        }
        __syncwarp();
        TOut* const ydst = static_cast<TOut*>(job.y) + head_off + (size_t)t0 * args.sT + q * 32 + lane;
        const auto put = [&](int t, uint32_t w, float f) {
          const uint32_t uw = __shfl_sync(0xffffffffu, upair[t >> 1], ((t & 1) << 4) + (lane >> 1));
          const float y = __uint_as_float(w) * f * __uint_as_float((lane & 1) ? (uw & 0xffff0000u) : (uw << 16));
          store_below(ydst, stride, t, y, rows);
          if (GATED == 2) store_below(dst, stride, t, __uint_as_float(w), rows);
        };
        tmem_ld_wait();
#pragma unroll
        for (int p = 0; p < 4; ++p) {  // 16 tokens at a time
#pragma unroll
          for (int t4 = 0; t4 < 16; t4 += 4) {
            const float4 f = *reinterpret_cast<const float4*>(&factor[16 * p + t4]);
            const int x = 16 * (p % 2) + t4, t = 16 * p + t4;
            put(t, o[x], f.x);
            put(t + 1, o[x + 1], f.y);
            put(t + 2, o[x + 2], f.z);
            put(t + 3, o[x + 3], f.w);
          }
          if (p < 2) {  // the next 16 tokens into the registers of these
            tmem_ld_x16(colO + 32 + 16 * p, *reinterpret_cast<uint32_t(*)[16]>(&o[16 * p]));
            tmem_ld_wait();
          }
          if (p == 1) {
            tc_fence_before_sync();
            WARP_ARRIVE(W_M2_OK);  // M2 of the next block may overwrite O
          }
        }
      } else {
#pragma unroll 1
        for (int pc = 0; pc < 2; ++pc) {  // 32 tokens at a time
          uint32_t w[32];
          tmem_ld_x32(colO + pc * 32, w);
          tmem_ld_wait();
          if (pc == 1) {
            tc_fence_before_sync();
            WARP_ARRIVE(W_M2_OK);  // M2 of the next block may overwrite O
          }
          const int here = rows - pc * 32;
          if (here >= 32) {
#pragma unroll
            for (int x = 0; x < 32; ++x) store_at(dst, stride, x, __uint_as_float(w[x]));
          } else {
#pragma unroll
            for (int x = 0; x < 32; ++x)
              if (x < here) store_at(dst, stride, x, __uint_as_float(w[x]));
          }
          dst += 32 * args.sT;
        }
      }
    }
  }

teardown:
  if (EARLY && args.follows != FOLLOWS_ANY) grid_dep_wait();  // (a launch is complete only when those before it are)
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

template <bool REV, typename TOut, int GATED>
cudaError_t launch_walk_t(const TcMaps& m0, const TcMaps& m1, const TcArgs& ta, const DecayTable& tab, cudaStream_t stream) {
  const size_t smem = sizeof(WSmem<REV>) + 1024;
  static_assert(sizeof(WSmem<REV>) + 1024 <= 232448, "shared memory of one SM");
  const bool early = early_walks(ta.BH, ta.nseg, ta.seg_len);
  auto kern = early ? tc_walk_kernel<REV, TOut, GATED, true> : tc_walk_kernel<REV, TOut, GATED, false>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  KernelTimer timer(ta.njobs == 2 ? K_WALK_PAIR : K_WALK, stream);
  err = launch_kernel(early, kern, dim3((unsigned)(ta.BH * ta.nseg * ta.njobs)), dim3(W_THREADS), smem, stream, 1, m0, m1, ta, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}
