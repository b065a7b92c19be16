// Segment states (included by la_tc.cu, inside its anonymous namespace, after the helpers): per (batch*head,
// segment) the local state sum_t decay-to-segment-edge * b_t c_t^T, which the walk chains into the state entering each
// segment.
//
// As in the walk the product is turned, dZ^T [e, d] = fc^T b with fc = diag(f) c as the A operand in tensor memory (lane =
// value column), so that one thread block makes all 128 columns, nothing formed on chip goes through shared memory, and the
// result leaves as whole 128-byte lines.  A block whose every token weight is exactly zero in fp32 (exp2f underflows past
// the smallest subnormal) adds exactly nothing and is not loaded: a decaying head reads only the 160 / s2 + 256 tokens next
// to the segment's edge.  What is left is bound by its longest thread block, a slowly decaying head that walks whole
// segments, while most others have two or three blocks to do.  So the blocks of such a segment are shared out over the
// thread blocks of a cluster, which add up their parts through distributed shared memory in a fixed order; the other
// segments fill whole clusters too, one thread block each, without talking to one another.
// A thread block's own start and end (set-up 1.1 us, first tile from HBM 1.3 to 1.7, result 1.2) take as long as four
// blocks, so two of them share an SM: pieces of 64 tokens, three load stages (96 KB) and half of tensor memory each.
//
// Warps: 0 TMA producer, 1 MMA issuer, 4-19 workers (32 value columns x 32 tokens of fc of every other piece each).

// D = 64: the hi terms of fc are in lanes 0 .. 63 and the lo terms in lanes 64 .. 127, one product of 64 columns for both, whose
// halves are added up on the way out.  A piece is 16 KB, so that six stages hold as much as three.

constexpr int S_THREADS = 640;
constexpr uint32_t S_TMEM_COLS = 256;
constexpr uint32_t SCOL_Z = 0, SCOL_F = 128;  // two fc buffers of 64 columns (hi, lo), or four of 32 (hi alone, or D = 64)

// Which (batch, head, segment) a thread block works on: `order` has the slowly decaying heads first, so that the longest
// chains start first (B = 1, H = 32, N = 65536, chains of 57 blocks: 118 us with the heads in their own order, 97 in this
// one).  Clusters take the segments of the `n_shared` heads at its front, one per cluster, then those of the other heads,
// one per thread block.
struct StatePlan {
  int n_shared, cluster;     // clusters share the segments of the first n_shared heads
  int nseg_used, seg_first;  // segments seg_first .. seg_first + nseg_used - 1 of the args.nseg
  unsigned char order[LA_MAX_H];
};

// The loads of piece p arrive on barrier p % FULLS: all pieces of one barrier belong to the same group of workers, which
// waits for no others.  (With a barrier per stage a group had to see the other's pieces go by, and nothing kept a stage from
// being loaded again, twice, before a warp that came late had looked; it then waited until its budget ran out.)
template <int D>
struct SBar {
  static constexpr int STAGES = D == 128 ? 3 : 6, FULLS = D == 128 ? 2 * STAGES : STAGES;
  static constexpr int FULL0 = 0, FREE0 = FULL0 + FULLS, FC_READY0 = FREE0 + STAGES, FC_FREE0 = FC_READY0 + 4, DONE = FC_FREE0 + 4,
                       DRAIN = DONE + 1, NUM = DRAIN + 1;
};

template <int D>
struct alignas(1024) SSmem {
  uint64_t bars[SBar<D>::NUM];
  uint32_t tmem_slot;
  int abort;
  struct alignas(1024) Stage {
    __nv_bfloat16 b[D / 64][64 * 64], c[D / 64][64 * 64];
  } stage[SBar<D>::STAGES];
};
static_assert(3 * sizeof(SSmem<128>::Stage) >= 128 * 128 * 4 && 6 * sizeof(SSmem<64>::Stage) >= 2 * 64 * 64 * 4, "a part of the state fits the stages");

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t saddr, uint32_t rank) {
  uint32_t a;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}

template <bool REV, int D>
__global__ void __launch_bounds__(S_THREADS, 2)
tc_state_kernel(const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_c,
                const __grid_constant__ TcArgs args, const __grid_constant__ StatePlan plan, const __grid_constant__ DecayTable tab) {
  extern __shared__ unsigned char smem_raw[];
  using SB = SBar<D>;
  constexpr int S_STAGES = SB::STAGES, S_FULLS = SB::FULLS, S_FULL0 = SB::FULL0, S_FREE0 = SB::FREE0, S_FC_READY0 = SB::FC_READY0,
                S_FC_FREE0 = SB::FC_FREE0, S_DONE = SB::DONE, S_DRAIN = SB::DRAIN, S_NUM_BARS = SB::NUM;
  constexpr int PANELS = D / 64;
  SSmem<D>& sm = *reinterpret_cast<SSmem<D>*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (args.seq_start) grid_dep_wait();  // the tables of a packed batch

  // ---- which segment, and which of its pieces ----
  const int cid = blockIdx.x / plan.cluster, rank = blockIdx.x % plan.cluster;
  const int B = args.BH / args.H;
  const int n_shared = plan.n_shared * B * plan.nseg_used;
  const bool shared = cid < n_shared;
  const int unit = shared ? cid : (cid - n_shared) * plan.cluster + rank + n_shared;
  if (unit >= args.BH * plan.nseg_used) return;
  const int h = plan.order[unit / (B * plan.nseg_used)];
  const int seg = plan.seg_first + unit % plan.nseg_used;
  int b = unit / plan.nseg_used % B;
  if (args.seq_order) b = args.seq_order[b];
  const int bh = b * args.H + h;
  const int n_tok = args.seq_len ? args.seq_len[b] : args.N;
  const int tok0 = args.seq_start ? args.seq_start[b] : 0;
  const int bb = args.seq_start ? 0 : b;
  const int bf = args.fold && bb >= args.fold ? bb - args.fold : bb;  // of an operand that is shared
  const int bat_b = args.job[0].shared & SHARED_B ? bf : bb, bat_c = args.job[0].shared & SHARED_C ? bf : bb;
  const int seg_t0 = seg * args.seg_len, seg_t1 = min(n_tok, seg_t0 + args.seg_len);
  if (seg_t0 >= n_tok) return;  // (all thread blocks of a cluster that shares a segment alike)
  const float s2 = (float)tab.s2[h];
  const bool split_c = (args.precision & 4) != 0 && s2 != 0.f;  // lambda == 1: the lo term is identically zero
  const int nf = D == 128 && split_c ? 2 : 4, fcols = D == 128 && split_c ? 64 : 32;  // fc buffers, and their columns
  int first = 0, count = (seg_t1 - seg_t0 + 127) >> 7;
  if (s2 > 0.f) {
    // blocks whose nearest token is within 160 / s2 + 128 tokens of the edge (the margin makes the skipped weights zero
    // whatever the rounding of this bound)
    const float reach = 160.f / s2;
    if (REV) {
      count = max(1, (int)fminf(ceilf((reach - 1.f) * (1.f / 128.f)) + 2.f, (float)count));
    } else {
      const float x = ((float)(seg_t1 - seg_t0) - reach) * (1.f / 128.f);  // blocks before the reach
      first = max(0, min(count - 1, (int)floorf(x - 1.f)));
      count -= first;
    }
  }
  first *= 2;  // in pieces of 64 tokens from here on
  count = min(2 * count, ((seg_t1 - seg_t0 + 63) >> 6) - first);
  if (shared) {
    const int lo = count * rank / plan.cluster, hi = count * (rank + 1) / plan.cluster;
    first += lo;
    count = hi - lo;  // may be 0
  }

  // Pieces are taken towards the edge that the state leaves through, so that the small products come first: away from it the
  // error of a lambda = 0.9995 state doubles (3.6e-6 to 7.7e-6).  The two pieces of a block keep the order of its tokens.
  const auto piece = [&](int it) {
    if (!REV) return first + it;
    const int p = first + count - 1 - it, mate = p ^ 1;
    return mate >= first && mate < first + count ? mate : p;
  };

  if (tid == 0) {
    for (int i = 0; i < S_NUM_BARS; ++i) mbar_init(&sm.bars[i], (i >= S_FC_READY0 && i < S_FC_FREE0) ? 8 : 1);
    sm.abort = 0;
    fence_mbar_init();
    tma_prefetch_desc(&map_b);
    tma_prefetch_desc(&map_c);
  }
  if (warp == 1) {
    grid_dep_wait();  // (see Follows)
    tmem_alloc(&sm.tmem_slot, S_TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sm.tmem_slot;
  grid_dep_wait();
  grid_dep_launch();

  if (warp == 0) {
    // ------------------------------------ TMA producer ------------------------------------
    if (lane == 0) {
      int armed = 0;
      for (int it = 0, s = 0, phase = 0, f = 0; it < count; ++it) {
        if (it >= S_STAGES) TC_WAIT_TO(producer_done, S_FREE0 + s, phase ^ 1, 31);
        const int t = tok0 + seg_t0 + piece(it) * 64;
        uint64_t* bar = &sm.bars[S_FULL0 + f];
        if (++f == S_FULLS) f = 0;
        mbar_arrive_expect_tx(bar, PANELS * 16384);
#pragma unroll
        for (int x = 0; x < PANELS; ++x) tma_load_4d(&sm.stage[s].c[x][0], &map_c, bar, x * 64, t, h, bat_c);
#pragma unroll
        for (int x = 0; x < PANELS; ++x) tma_load_4d(&sm.stage[s].b[x][0], &map_b, bar, x * 64, t, h, bat_b);
        armed = it + 1;
        if (++s == S_STAGES) s = 0, phase ^= 1;
      }
    producer_done:
      if (sm.abort)  // nothing may be in flight when the block exits
        for (int k = 0; k < S_STAGES; ++k)
          if (armed - 1 - k >= 0) drain_wait(&sm.bars[S_FULL0 + (armed - 1 - k) % S_FULLS], ((armed - 1 - k) / S_FULLS) & 1);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------ MMA issuer ------------------------------------
    constexpr uint32_t ID_KN = umma_idesc_bf16(128, D, false, true);  // tensor-memory A x MN-major B
    constexpr uint32_t HI = UMMA_DESC_HI_SBO1024;
    constexpr uint32_t STAGE = (uint32_t)(sizeof(typename SSmem<D>::Stage) >> 4);
    const uint32_t go = elect_one();
    const uint32_t b0 = umma_desc_lo(smem_u32(&sm.stage[0].b[0][0]), 8192);
    for (int it = 0, s = 0, u = 0, phase = 0, f = 0, fphase = 0; it < count; ++it) {
      TC_WAIT_WARP_TO(mma_done, S_FULL0 + u, phase, 32);
      TC_WAIT_WARP_TO(mma_done, S_FC_READY0 + f, fphase, 33);
      tc_fence_after_sync();
      const uint32_t fcol = tmem + SCOL_F + f * fcols;
      umma_group_tsd4<false>(tmem + SCOL_Z, fcol, b0 + s * STAGE, HI, ID_KN, it > 0 ? 1u : 0u, go);
      if (D == 128 && split_c) umma_group_tsd4<false>(tmem + SCOL_Z, fcol + 32, b0 + s * STAGE, HI, ID_KN, 1, go);
      umma_commit_if(&sm.bars[S_FREE0 + s], go);
      umma_commit_if(&sm.bars[S_FC_FREE0 + f], go);
      if (++s == S_STAGES) s = 0;
      if (++u == S_FULLS) u = 0, phase ^= 1;
      if (++f == nf) f = 0, fphase ^= 1;
    }
    umma_commit_if(&sm.bars[S_DONE], go);
  mma_done:
    if (sm.abort) {
      umma_commit_if(&sm.bars[S_DRAIN], go);
      drain_wait(&sm.bars[S_DRAIN], 0);
    }
  } else if (warp >= 4) {
    // ------------------------------------ workers ------------------------------------
    const int q = warp & 3, w4 = (warp - 4) >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    // The sixteen warps take turns in two groups, 32 tokens of a piece per warp, so that two pieces are under way at a time.
    // Where lambda = 1 fc is c and goes to tensor memory as it is: this is the head with the longest chains, and a chain is
    // bound by the instructions between two pieces (57 blocks in one thread block: 66 us through split2, 45 us this way; the
    // shape above: 97 and 83).
    const int group = w4 >> 1;
    // lane l points ldmatrix at token row (w4 & 1) * 32 + (l >> 4) * 8 + (l & 7), value columns q * 32 (D = 64:
    // (q & 1) * 32) + ((l >> 3) & 1) * 8
    const bool lo_part = D == 64 && q >= 2;
    const uint32_t unit0 = (uint32_t)((D == 128 ? (q >> 1) * 8192 : 0) + ((w4 & 1) * 32 + ((lane >> 4) << 3) + (lane & 7)) * 128 +
                                      ((((q & 1) * 4 + ((lane >> 3) & 1)) ^ (lane & 7)) << 4));
    for (int it = group, u = group, phase = 0, fb = group, fphase = 0; it < count; it += 2) {
      const int st = u < S_STAGES ? u : u - S_STAGES;
      TC_WAIT_WARP(S_FULL0 + u, phase, 34);
      u += 2;
      if (u >= S_FULLS) u -= S_FULLS, phase ^= 1;
      if (it >= nf) TC_WAIT_WARP(S_FC_FREE0 + fb, fphase ^ 1, 35);
      tc_fence_after_sync();
      const int own = seg_t1 - (seg_t0 + piece(it) * 64);  // tokens of this piece that are the segment's
      if (args.seq_start && own < 64) {
        // packed batch: what follows is another sequence's and must not come through its zero weight either (0 * inf)
        for (int x = own * 8 + ((w4 & 1) * 4 + q) * 32 + lane; x < 512; x += 256)
#pragma unroll
          for (int n = 0; n < PANELS; ++n) reinterpret_cast<uint4*>(sm.stage[st].b[n])[x] = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async_smem();
      }
      if (lo_part && !split_c) {
        WARP_ARRIVE(S_FC_READY0 + fb);
        fb += 2;
        if (fb >= nf) fb -= nf, fphase ^= 1;
        continue;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {  // 16 tokens at a time
        uint32_t raw[8];             // [16 value columns][8 tokens][8 value columns]
        const uint32_t ctile = smem_u32(&sm.stage[st].c[0][0]) + unit0 + k * 2048;
#pragma unroll
        for (int g = 0; g < 2; ++g)
          ldmatrix_x4_trans(ctile ^ (g << 5), raw[4 * g], raw[4 * g + 1], raw[4 * g + 2], raw[4 * g + 3]);
        const uint32_t colF = lane_addr + SCOL_F + fb * fcols + (w4 & 1) * 16 + k * 8;
        const int p0 = seg_t0 + piece(it) * 64;
        if (s2 == 0.f && p0 + 64 <= seg_t1) {
          tmem_st_16x128b_x2(colF, *reinterpret_cast<uint32_t(*)[4]>(&raw[0]));
          tmem_st_16x128b_x2(colF + (16u << 16), *reinterpret_cast<uint32_t(*)[4]>(&raw[4]));
          continue;
        }
        const int t0 = p0 + (w4 & 1) * 32 + k * 16 + 2 * (lane & 3);
        float f[4];  // decay from this thread's tokens to the edge that the state leaves the segment through
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int t = t0 + 8 * (o >> 1) + (o & 1);
          f[o] = t < seg_t1 ? exp2f(-s2 * (float)(REV ? t - seg_t0 + 1 : seg_t1 - 1 - t)) : 0.f;
        }
        if (own < 64) {
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            const int t = t0 + 8 * ((x >> 1) & 1);
            raw[x] &= (t < seg_t1 ? 0xffffu : 0u) | (t + 1 < seg_t1 ? 0xffff0000u : 0u);
          }
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint32_t hh[4], ll[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const uint32_t w = raw[4 * g + x];
            split2(f2_pack(__uint_as_float(w << 16) * f[(x >> 1) * 2], __uint_as_float(w & 0xffff0000u) * f[(x >> 1) * 2 + 1]),
                   hh[x], ll[x]);
          }
          const uint32_t at = colF + ((uint32_t)(g * 16) << 16);
          if (D == 64) {
            tmem_st_16x128b_x2(at, lo_part ? ll : hh);
          } else {
            tmem_st_16x128b_x2(at, hh);
            if (split_c) tmem_st_16x128b_x2(at + 32, ll);
          }
        }
      }
      tmem_st_wait();
      tc_fence_before_sync();
      WARP_ARRIVE(S_FC_READY0 + fb);
      fb += 2;
      if (fb >= nf) fb -= nf, fphase ^= 1;
    }
    // ---- result: value column q * 32 + lane (D = 64: that of the hi or the lo half), features w4 * D / 4 .. ----
    constexpr int PER = D / 4;
    uint32_t z[PER];
    if (count > 0) {
      TC_WAIT_WARP(S_DONE, 0, 36);
      tc_fence_after_sync();
#pragma unroll
      for (int x = 0; x < PER; x += 16) tmem_ld_x16(lane_addr + SCOL_Z + w4 * PER + x, *reinterpret_cast<uint32_t(*)[16]>(&z[x]));
      tmem_ld_wait();
      tc_fence_before_sync();
    }
    if (count == 0 || (lo_part && !split_c)) {
#pragma unroll
      for (int x = 0; x < PER; ++x) z[x] = 0u;
    }
    // (every load has been read)
    if (D == 64) {
      float* part = reinterpret_cast<float*>(&sm.stage[0]) + (lo_part ? D * D : 0) + (w4 * PER) * D + (q & 1) * 32 + lane;
#pragma unroll
      for (int x = 0; x < PER; ++x) part[x * D] = __uint_as_float(z[x]);
    } else {
      float* dst = args.local_out + ((size_t)bh * args.nseg + seg) * (D * D) + (size_t)(w4 * PER) * D + q * 32 + lane;
      float* part = reinterpret_cast<float*>(&sm.stage[0]) + (w4 * PER) * D + q * 32 + lane;
#pragma unroll
      for (int x = 0; x < PER; ++x) {
        if (shared) part[x * D] = __uint_as_float(z[x]);
        else dst[x * D] = __uint_as_float(z[x]);
      }
    }
  }

teardown:
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, S_TMEM_COLS);
  if (shared || D == 64) {
    // each thread block of the cluster adds up its share of the parts, in rank order, the hi halves first
    const int ranks = shared ? plan.cluster : 1, first_rank = shared ? rank : 0;
    if (shared) cluster_sync();
    const int per = D * D / 4 / ranks;  // float4 groups of the state per thread block
    float4* out = reinterpret_cast<float4*>(args.local_out + ((size_t)bh * args.nseg + seg) * (D * D));
    for (int i = first_rank * per + tid; i < (first_rank + 1) * per; i += S_THREADS) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int half = 0; half < (D == 64 ? 2 : 1); ++half) {
        const uint32_t at = smem_u32(&sm.stage[0]) + (half * (D * D / 4) + i) * 16;
        if (!shared) {
          const float4 x = reinterpret_cast<const float4*>(&sm.stage[0])[half * (D * D / 4) + i];
          v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
          continue;
        }
        float4 x[8];  // all loads first: one by one they take 700 clocks each
#pragma unroll
        for (int r = 0; r < 8; ++r) x[r] = r < plan.cluster ? ld_cluster_f4(at, (uint32_t)r) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (half == 0) v = x[0];
        else v.x += x[0].x, v.y += x[0].y, v.z += x[0].z, v.w += x[0].w;
#pragma unroll
        for (int r = 1; r < 8; ++r) {
          v.x += x[r].x; v.y += x[r].y; v.z += x[r].z; v.w += x[r].w;
        }
      }
      out[i] = v;
    }
    if (shared) cluster_sync();  // nobody leaves while its part is being read
  }
}

// Splits the work: cluster size and the heads whose segments are shared, in units of one block (1.3 us).  A thread block
// costs its blocks plus 4.5 (start, end), in a cluster 7, 7.5 or 10, behind clusters 2 more; a launch costs its longest thread
// block (a quarter of the time that HBM is busy longer), the total over 200 (two thread blocks on an SM slow one
// another down), or the blocks read at 100 to a unit (HBM), whichever is the most, and a little of the first two.
// Measured with the cluster size forced, la_chunk_state, us unshared / 2 / 4 / 8: 32 heads x 777 19 / 18.5 / 16.4 /
// 22.5; 16 x 32768 38 / 31.5 / 38 / 66; 16 heads of lambda = 1 x 65536 97 / 102 / 117 / 129; the 7B-like shape 81 / 58 / 72 / 132.
// Segments of more than 32 blocks are shared by two at most.  A chain of products in one accumulator carries a rounding bias,
// 1.3e-5 of a lambda = 1 state after 57 blocks, and cutting it, which takes that away, moves the results of the 7B-like step:
// by 6e-6 in the 2-norm shared by two, by 7.4e-6 shared by four and eight (la_chunk_state there: 54 us and 45).
inline StatePlan make_state_plan(const TcArgs& ta, const DecayTable& tab, bool rev, bool all_segments) {
  StatePlan p{};
  p.nseg_used = all_segments ? ta.nseg : ta.nseg - 1;
  p.seg_first = (rev && !all_segments) ? 1 : 0;
  const int blocks = (ta.seg_len + 127) / 128;
  int keep[LA_MAX_H];
  for (int h = 0; h < ta.H; ++h) {
    const double reach = tab.s2[h] > 0.0 ? 160.0 / tab.s2[h] / 128.0 + 2.0 : 1e9;
    keep[h] = reach < blocks ? (int)reach + 1 : blocks;
    if (keep[h] > blocks) keep[h] = blocks;
  }
  const double units = (double)(ta.BH / ta.H) * p.nseg_used;
  double best = 1e30;
  int best_limit = 0;
  p.cluster = 1;
  for (int cl = 1; cl <= (blocks > 32 ? 2 : 8); cl *= 2) {
    const double around = cl == 2 ? 7.0 : cl == 4 ? 7.5 : 10.0;
    for (int limit = 2; limit <= 64; limit *= 2) {  // heads that keep more blocks than this are shared
      double total = 0.0, longest = 0.0, read = 0.0;
      for (int h = 0; h < ta.H; ++h) {
        const bool sh = cl > 1 && keep[h] > limit;
        const double t = sh ? (keep[h] + cl - 1) / cl + around : keep[h] + (cl > 1 ? 6.5 : 4.5);
        total += units * t * (sh ? cl : 1);
        read += units * keep[h];
        if (t > longest) longest = t;
      }
      read *= 0.01;
      longest += 0.25 * (read < longest ? read : longest);
      const double busy = longest > total / 200.0 ? longest : total / 200.0;
      const double cost = (busy > read ? busy : read) + 0.1 * busy;
      if (cost < best * (p.cluster == 1 ? 0.9 : 0.95)) {
        best = cost;
        best_limit = limit;
        p.cluster = cl;
      }
      if (cl == 1) break;
    }
  }
  for (int h = 0; h < ta.H; ++h) {
    int at = h;
    for (; at > 0 && keep[p.order[at - 1]] < keep[h]; --at) p.order[at] = p.order[at - 1];
    p.order[at] = (unsigned char)h;
    p.n_shared += p.cluster > 1 && keep[h] > best_limit;
  }
  return p;
}

template <bool REV, int D>
cudaError_t launch_state_t(const TcMaps& m, const TcArgs& ta, const DecayTable& tab, bool all_segments, cudaStream_t stream) {
  const size_t smem = sizeof(SSmem<D>) + 1024;
  static_assert(2 * (sizeof(SSmem<D>) + 2048) <= 233472, "two thread blocks in the shared memory of one SM");
  auto kern = tc_state_kernel<REV, D>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  const StatePlan plan = make_state_plan(ta, tab, REV, all_segments);
  const long shared_units = (long)plan.n_shared * (ta.BH / ta.H) * plan.nseg_used;
  const long other_units = (long)(ta.H - plan.n_shared) * (ta.BH / ta.H) * plan.nseg_used;
  const long clusters = shared_units + (other_units + plan.cluster - 1) / plan.cluster;
  KernelTimer timer(K_PREPASS, stream);
  err = launch_kernel(early_walks(ta.BH, ta.nseg, ta.seg_len), kern, dim3((unsigned)(clusters * plan.cluster)), dim3(S_THREADS), smem, stream, plan.cluster,
                      m.b, m.c, ta, plan, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}
