// fp32 CUDA-core kernels of the generic decayed linear-attention operator
// (see la_common.cuh for the block formulas).  They serve fp32 inputs and are the full-precision second opinion for the
// tensor-core kernels.  All arithmetic is fp32 FMA with fp32 accumulation; bf16 inputs are widened exactly on load.
//
// Tiles of C = 32 tokens.  simt_rows_kernel: segments of up to ROWS_MAX_SEG tokens, every row tile by itself.
// simt_walk_kernel: longer segments, one thread block of 256 threads per (batch*head, segment) that carries the Da x Ec state
// from block to block; shared memory holds the a/b/c tiles (a and b also transposed so that every inner loop reads consecutive
// addresses), the masked score tile and the state.
#include <algorithm>

#include "la_common.cuh"

namespace la {

namespace {

constexpr int C = 32;
constexpr int THREADS = 256;
constexpr int AP = C + 4;  // padded row length of the transposed tiles

template <int DA, int EC>
struct Smem {
  float aT[DA][AP];  // aT[k][i] = a[i][k]
  float bT[DA][AP];
  float b[C][DA];
  float c[C][EC];
  float pT[C][AP];  // pT[j][i] = masked score of (row i, column j)
  float Z[DA][EC];
  float dtab[C];     // lambda^n, n = 0..C-1
  float f_out[C];
  float f_state[C];
  float gamma;
};

template <typename TIn, int W>
__device__ __forceinline__ void load_tile_natural(float (*dst)[W], const TIn* src, long long row_stride, int rows_valid) {
  // dst[i][k] = src[i*row_stride + k] for i < rows_valid, else 0
  for (int idx = threadIdx.x; idx < C * W; idx += THREADS) {
    const int i = idx / W, k = idx % W;
    dst[i][k] = (i < rows_valid) ? to_f32<TIn>(src[(size_t)i * row_stride + k]) : 0.f;
  }
}

template <typename TIn, int W>
__device__ __forceinline__ void load_tile_transposed(float (*dstT)[AP], const TIn* src, long long row_stride,
                                                     int rows_valid) {
  for (int idx = threadIdx.x; idx < C * W; idx += THREADS) {
    const int i = idx / W, k = idx % W;
    dstT[k][i] = (i < rows_valid) ? to_f32<TIn>(src[(size_t)i * row_stride + k]) : 0.f;
  }
}

template <typename TIn, typename TOut, int DA, int EC, bool REV>
__global__ void __launch_bounds__(THREADS, 1)
simt_walk_kernel(const OpArgs args, const DecayTable tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<DA, EC>& sm = *reinterpret_cast<Smem<DA, EC>*>(smem_raw);

  const int tid = threadIdx.x;
  const int bh = blockIdx.x / args.nseg;
  const int seg = blockIdx.x % args.nseg;
  const double s2 = tab.s2[bh % args.H];
  const int seg_t0 = seg * args.seg_len;
  const int seg_t1 = min(args.N, seg_t0 + args.seg_len);
  const int nblk = (seg_t1 - seg_t0 + C - 1) / C;

  const size_t head_off = (size_t)(bh / args.H) * args.sB + (size_t)(bh % args.H) * args.sH;
  const long long sT = args.sT;  // elements between consecutive tokens
  const TIn* a = static_cast<const TIn*>(args.a) + head_off;
  const TIn* b = static_cast<const TIn*>(args.b) + head_off;
  const TIn* c = static_cast<const TIn*>(args.c) + head_off;
  TOut* out = static_cast<TOut*>(args.out) + head_off;

  // state entering this segment
  {
    const float* zin = args.entry ? args.entry + ((size_t)bh * args.nseg + seg) * DA * EC : nullptr;
    float* zf = &sm.Z[0][0];
    for (int idx = tid; idx < DA * EC; idx += THREADS) zf[idx] = zin ? zin[idx] : 0.f;
  }
  if (tid < C) sm.dtab[tid] = decay_pow_d(s2, (double)tid);

  for (int ib = 0; ib < nblk; ++ib) {
    const int blk = REV ? (nblk - 1 - ib) : ib;
    const int t0 = seg_t0 + blk * C;
    const int Cr = min(C, seg_t1 - t0);

    if (tid < C) {
      const int i = tid;
      if (!REV) {
        sm.f_out[i] = decay_pow_d(s2, (double)(i + 1));
        sm.f_state[i] = (i < Cr) ? decay_pow_d(s2, (double)(Cr - 1 - i)) : 0.f;
      } else {
        sm.f_out[i] = (i < Cr) ? decay_pow_d(s2, (double)(Cr - 1 - i)) : 0.f;
        sm.f_state[i] = decay_pow_d(s2, (double)(i + 1));
      }
      if (i == 0) sm.gamma = decay_pow_d(s2, (double)Cr);
    }
    load_tile_transposed<TIn, DA>(sm.aT, a + (size_t)t0 * sT, sT, Cr);
    load_tile_transposed<TIn, DA>(sm.bT, b + (size_t)t0 * sT, sT, Cr);
    load_tile_natural<TIn, DA>(sm.b, b + (size_t)t0 * sT, sT, Cr);
    load_tile_natural<TIn, EC>(sm.c, c + (size_t)t0 * sT, sT, Cr);
    __syncthreads();

    // (1) masked scores: pT[j][i] = (a_i . b_j) * D_ij
    {
      const int ty = tid / 16, tx = tid % 16;
      float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll 8
      for (int k = 0; k < DA; ++k) {
        const float a0 = sm.aT[k][2 * ty], a1 = sm.aT[k][2 * ty + 1];
        const float b0 = sm.bT[k][2 * tx], b1 = sm.bT[k][2 * tx + 1];
        acc[0][0] = fmaf(a0, b0, acc[0][0]);
        acc[0][1] = fmaf(a0, b1, acc[0][1]);
        acc[1][0] = fmaf(a1, b0, acc[1][0]);
        acc[1][1] = fmaf(a1, b1, acc[1][1]);
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const int i = 2 * ty + r, j = 2 * tx + cc;
          const int n = REV ? (j - i) : (i - j);
          // a select, not a multiply by zero: masked-out tokens can never leak
          sm.pT[j][i] = (n >= 0) ? acc[r][cc] * sm.dtab[n] : 0.f;
        }
    }
    __syncthreads();

    // (2)+(3) out = P c + diag(f_out) a Z
    {
      constexpr int EM = EC / 32;
      const int ty = tid / 32, tx = tid % 32;
      const int i0 = 4 * ty;
      float intra[4][EM], inter[4][EM];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int m = 0; m < EM; ++m) intra[r][m] = inter[r][m] = 0.f;
#pragma unroll 4
      for (int j = 0; j < C; ++j) {
        float p[4], cv[EM];
#pragma unroll
        for (int r = 0; r < 4; ++r) p[r] = sm.pT[j][i0 + r];
#pragma unroll
        for (int m = 0; m < EM; ++m) cv[m] = sm.c[j][tx + 32 * m];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int m = 0; m < EM; ++m) intra[r][m] = fmaf(p[r], cv[m], intra[r][m]);
      }
#pragma unroll 4
      for (int k = 0; k < DA; ++k) {
        float av[4], zv[EM];
#pragma unroll
        for (int r = 0; r < 4; ++r) av[r] = sm.aT[k][i0 + r];
#pragma unroll
        for (int m = 0; m < EM; ++m) zv[m] = sm.Z[k][tx + 32 * m];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int m = 0; m < EM; ++m) inter[r][m] = fmaf(av[r], zv[m], inter[r][m]);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + r;
        if (i < Cr) {
          const float f = sm.f_out[i];
#pragma unroll
          for (int m = 0; m < EM; ++m)
            out[(size_t)(t0 + i) * sT + tx + 32 * m] = from_f32<TOut>(fmaf(f, inter[r][m], intra[r][m]));
        }
      }
    }
    __syncthreads();

    // (4) Z <- Gamma Z + b^T diag(f_state) c
    {
      constexpr int RK = DA / 16, RE = EC / 16;
      const int ty = tid / 16, tx = tid % 16;
      float acc[RK][RE];
#pragma unroll
      for (int r = 0; r < RK; ++r)
#pragma unroll
        for (int m = 0; m < RE; ++m) acc[r][m] = 0.f;
#pragma unroll 2
      for (int j = 0; j < C; ++j) {
        float bv[RK], cv[RE];
        const float f = sm.f_state[j];
#pragma unroll
        for (int r = 0; r < RK; ++r) bv[r] = sm.b[j][ty + 16 * r];
#pragma unroll
        for (int m = 0; m < RE; ++m) cv[m] = f * sm.c[j][tx + 16 * m];
#pragma unroll
        for (int r = 0; r < RK; ++r)
#pragma unroll
          for (int m = 0; m < RE; ++m) acc[r][m] = fmaf(bv[r], cv[m], acc[r][m]);
      }
      const float g = sm.gamma;
#pragma unroll
      for (int r = 0; r < RK; ++r)
#pragma unroll
        for (int m = 0; m < RE; ++m) {
          float& z = sm.Z[ty + 16 * r][tx + 16 * m];
          z = fmaf(g, z, acc[r][m]);
        }
    }
    __syncthreads();
  }

  const bool last_processed = REV ? (seg == 0) : (seg == args.nseg - 1);
  if (args.final_out && last_processed) {
    float* dst = args.final_out + (size_t)bh * DA * EC;
    const float* zf = &sm.Z[0][0];
    for (int idx = tid; idx < DA * EC; idx += THREADS) dst[idx] = zf[idx];
  }
}

// Segment-local state: sum over the segment's tokens of decay-to-segment-edge * b_t c_t^T.
//   forward: edge = last token of the segment, factor lambda^(t1-1-t)
//   reverse: edge = first token, in the gauge the reverse walk carries: lambda^(t-t0+1)
template <typename TIn, int DA, int EC>
struct PreSmem {
  float b[C][DA];
  float c[C][EC];
  float f_state[C];
};

template <typename TIn, int DA, int EC, bool REV>
__global__ void __launch_bounds__(THREADS, 2)
simt_prepass_kernel(const OpArgs args, const DecayTable tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PreSmem<TIn, DA, EC>& sm = *reinterpret_cast<PreSmem<TIn, DA, EC>*>(smem_raw);
  const int tid = threadIdx.x;
  const int bh = blockIdx.x / args.nseg;
  const int seg = blockIdx.x % args.nseg;
  const double s2 = tab.s2[bh % args.H];
  const int seg_t0 = seg * args.seg_len;
  const int seg_t1 = min(args.N, seg_t0 + args.seg_len);
  const int nblk = (seg_t1 - seg_t0 + C - 1) / C;
  const size_t head_off = (size_t)(bh / args.H) * args.sB + (size_t)(bh % args.H) * args.sH;
  const long long sT = args.sT;
  const TIn* b = static_cast<const TIn*>(args.b) + head_off;
  const TIn* c = static_cast<const TIn*>(args.c) + head_off;

  constexpr int RK = DA / 16, RE = EC / 16;
  const int ty = tid / 16, tx = tid % 16;
  float acc[RK][RE];
#pragma unroll
  for (int r = 0; r < RK; ++r)
#pragma unroll
    for (int m = 0; m < RE; ++m) acc[r][m] = 0.f;

  for (int blk = 0; blk < nblk; ++blk) {
    const int t0 = seg_t0 + blk * C;
    const int Cr = min(C, seg_t1 - t0);
    if (tid < C) {
      const int t = t0 + tid;
      float f = 0.f;
      if (tid < Cr) f = REV ? decay_pow_d(s2, (double)(t - seg_t0 + 1)) : decay_pow_d(s2, (double)(seg_t1 - 1 - t));
      sm.f_state[tid] = f;
    }
    load_tile_natural<TIn, DA>(sm.b, b + (size_t)t0 * sT, sT, Cr);
    load_tile_natural<TIn, EC>(sm.c, c + (size_t)t0 * sT, sT, Cr);
    __syncthreads();
#pragma unroll 2
    for (int j = 0; j < C; ++j) {
      float bv[RK], cv[RE];
      const float f = sm.f_state[j];
#pragma unroll
      for (int r = 0; r < RK; ++r) bv[r] = sm.b[j][ty + 16 * r];
#pragma unroll
      for (int m = 0; m < RE; ++m) cv[m] = f * sm.c[j][tx + 16 * m];
#pragma unroll
      for (int r = 0; r < RK; ++r)
#pragma unroll
        for (int m = 0; m < RE; ++m) acc[r][m] = fmaf(bv[r], cv[m], acc[r][m]);
    }
    __syncthreads();
  }
  float* dst = args.local_out + ((size_t)bh * args.nseg + seg) * DA * EC;
#pragma unroll
  for (int r = 0; r < RK; ++r)
#pragma unroll
    for (int m = 0; m < RE; ++m) dst[(size_t)(ty + 16 * r) * EC + tx + 16 * m] = acc[r][m];
}

// Turns segment-local states into the state entering each segment, in place:
//   forward: x_0 = Z_in, x_{p+1} = lambda^(L_p) x_p + local_p
//   reverse: x_{last} = Z_in, x_{p-1} = lambda^(L_p) x_p + local_p
// One thread block per 32x32 tile of one (batch*head) state; each thread carries four elements
// across the short sequential walk over segments.  The optional transposed copy goes through a
// shared-memory tile so that both copies are written with coalesced stores.
constexpr int SCAN_MAX_SEG = 1024;
__global__ void __launch_bounds__(256) scan_kernel(const ScanArgs args, const DecayTable tab) {
  __shared__ float gamma[SCAN_MAX_SEG];
  __shared__ float tile[32][33];
  grid_dep_wait();
  grid_dep_launch();
  const int Da = args.Da, Ec = args.Ec, DE = Da * Ec;
  const int bh = blockIdx.x;
  const int tiles_y = Ec / 32;
  const int x0 = (blockIdx.y / tiles_y) * 32, y0 = (blockIdx.y % tiles_y) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  const double s2 = tab.s2[bh % args.H];
  const int n_tok = args.N, nseg = args.nseg;
  for (int p = threadIdx.x; p < nseg; p += 256) {
    const int L = min(n_tok, (p + 1) * args.seg_len) - p * args.seg_len;
    gamma[p] = decay_pow_d(s2, (double)L);
  }
  float z[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int x = x0 + ty + 8 * k, y = y0 + tx;
    z[k] = 0.f;
    if (args.z_in) z[k] = args.z_in[(size_t)bh * DE + (args.z_in_transposed ? (y * Da + x) : (x * Ec + y))];
  }
  __syncthreads();
  // the local state of a segment is fetched one step ahead of its use: the chain over segments is
  // sequential, and this keeps one global-memory round trip out of every step
  auto seg_of = [&](int ip) { return args.reverse ? (nseg - 1 - ip) : ip; };
  float loc[4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    loc[k] = (nseg > 1) ? args.buf[((size_t)bh * args.nseg + seg_of(0)) * DE + (size_t)(x0 + ty + 8 * k) * Ec + y0 + tx] : 0.f;
  for (int ip = 0; ip < nseg; ++ip) {
    const int p = seg_of(ip);
    const size_t off = ((size_t)bh * args.nseg + p) * DE;
    const bool more = (ip + 1 < nseg);
    float nxt[4] = {0.f, 0.f, 0.f, 0.f};
    if (ip + 2 < nseg) {
      const size_t offn = ((size_t)bh * args.nseg + seg_of(ip + 1)) * DE;
#pragma unroll
      for (int k = 0; k < 4; ++k) nxt[k] = args.buf[offn + (size_t)(x0 + ty + 8 * k) * Ec + y0 + tx];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) args.buf[off + (size_t)(x0 + ty + 8 * k) * Ec + y0 + tx] = z[k];
    if (args.buf_t) {
#pragma unroll
      for (int k = 0; k < 4; ++k) tile[ty + 8 * k][tx] = z[k];
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 4; ++k)
        args.buf_t[off + (size_t)(y0 + ty + 8 * k) * Da + x0 + tx] = tile[tx][ty + 8 * k];
      __syncthreads();
    }
    if (more) {
      const float g = gamma[p];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        z[k] = fmaf(g, z[k], loc[k]);
        loc[k] = nxt[k];
      }
    }
  }
}

// The walk of segments of at most ROWS_MAX_SEG tokens without a chain of blocks: out = P c over the whole segment plus
// diag(f_out) a Z, each 32-row tile of it by a thread block of its own, and the final state in 32-row tiles too.  All of it
// is one loop, acc[32, EC] += w[j, 32]^T t[j, EC] over 32-row tiles t: rows of c with w the masked scores, rows of Z with w
// the decayed a, or (final state) rows of c with w the decayed b.
// A walk that carries the state from block to block is bound by that chain where it has few heads: 8 us a block at d = 64
// with two thread blocks on the chip.  Here the work grows with the square of the segment, but all tiles run at once, and the
// walks of a launch do too (B = 1, H = 2, N = 256, d = 64 in fp32, forward plus backward: 240 us before, 38 now; with N = 2048
// and 128-token segments 1155 and 81).
// 128 threads; at d = 128 57 KB and 168 registers, which let three thread blocks share an SM; the next tiles are loaded into
// registers while the present ones are multiplied.
//
// The tiles that a thread block adds up are shared out over G groups of 128 threads, each with its own pair of tiles in shared
// memory, whose sums meet at the end: with one group a tile costs 4400 clocks, a warp per scheduler waiting for its own loads.
// Where thread blocks fill the chip several times over, groups only add their meeting (rows_shared).
constexpr int ROWS_THREADS = 128;  // of a group
constexpr int ROWS_MAX_JOBS = 3;
static_assert(ROWS_MAX_SEG % C == 0, "whole tiles");

struct RowsArgs {
  OpArgs job[ROWS_MAX_JOBS];
  int first_block[ROWS_MAX_JOBS + 1];  // thread blocks of job j: first_block[j] .. first_block[j + 1] - 1
  int units[ROWS_MAX_JOBS];            // how many of them make rows; the others make states
};

template <int D, int G>
struct RowsSmem {
  float a[C][D + 4];   // rows of a (states: unused)
  struct Group {
    float b[C][D + 4];
    float t[C][D];     // rows of c or Z
    float w[C][AP];    // w[j][i]
  } group[G];
  float dtab[ROWS_MAX_SEG + 1];  // lambda^n
};

// 32 rows of D values into registers, 16 bytes (fp32) at a time; rows past `valid` are zero.
template <typename TIn, int D>
__device__ __forceinline__ void fetch_tile(float4 (&x)[D / 16], const TIn* src, long long row_stride, int valid, int tid) {
#pragma unroll
  for (int n = 0; n < D / 16; ++n) {
    const int idx = tid + n * ROWS_THREADS, row = idx / (D / 4), col = idx % (D / 4) * 4;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (row < valid) Vec4<TIn>::load(src + (size_t)row * row_stride + col, v);
    x[n] = make_float4(v[0], v[1], v[2], v[3]);
  }
}
template <int D, int W>
__device__ __forceinline__ void put_tile(float (*dst)[W], const float4 (&x)[D / 16], int tid) {
#pragma unroll
  for (int n = 0; n < D / 16; ++n) {
    const int idx = tid + n * ROWS_THREADS;
    *reinterpret_cast<float4*>(&dst[idx / (D / 4)][idx % (D / 4) * 4]) = x[n];
  }
}
template <int G>
__device__ __forceinline__ void group_sync(int grp) {
  if (G == 1) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(ROWS_THREADS) : "memory");
}

template <typename TIn, typename TOut, int D, int G>
__global__ void __launch_bounds__(ROWS_THREADS * G)
simt_rows_kernel(const __grid_constant__ RowsArgs all, const __grid_constant__ DecayTable tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RowsSmem<D, G>& sm = *reinterpret_cast<RowsSmem<D, G>*>(smem_raw);
  grid_dep_wait();
  grid_dep_launch();
  const int grp = threadIdx.x / ROWS_THREADS, tid = threadIdx.x % ROWS_THREADS;
  typename RowsSmem<D, G>::Group& gm = sm.group[grp];
  int jb = 0;
  while (jb + 1 < ROWS_MAX_JOBS && (int)blockIdx.x >= all.first_block[jb + 1]) ++jb;
  const OpArgs& args = all.job[jb];
  int unit = (int)blockIdx.x - all.first_block[jb];
  const bool rev = args.reverse != 0;
  const bool state = unit >= all.units[jb];  // the state leaving the sequence, or (local_out) every segment's local state
  const int per_seg = (args.seg_len + C - 1) / C;
  int bh, seg, tile;
  if (state) {
    unit -= all.units[jb];
    tile = unit % (D / C);
    bh = unit / (D / C);
    seg = rev ? 0 : args.nseg - 1;
    if (args.local_out) {
      seg = bh % args.nseg;
      bh /= args.nseg;
    }
  } else {
    // the row tiles with the most tiles to add up first
    tile = unit / (args.BH * args.nseg);
    if (!rev) tile = per_seg - 1 - tile;
    seg = unit % args.nseg;
    bh = unit / args.nseg % args.BH;
  }
  const double s2 = tab.s2[bh % args.H];
  const int seg_t0 = seg * args.seg_len;
  const int L = min(args.N, seg_t0 + args.seg_len) - seg_t0;
  if (!state && tile * C >= L) return;

  const size_t head_off = (size_t)(bh / args.H) * args.sB + (size_t)(bh % args.H) * args.sH + (size_t)seg_t0 * args.sT;
  const long long sT = args.sT;
  const TIn* b = static_cast<const TIn*>(args.b) + head_off;
  const TIn* c = static_cast<const TIn*>(args.c) + head_off;
  const float* Z = args.entry ? args.entry + ((size_t)bh * args.nseg + seg) * D * D : nullptr;
  const int ntile = (L + C - 1) / C;
  // tiles of c to add up: the row tile's own first and then away from it; for the state towards the segment's edge
  const int step = (rev != state) ? 1 : -1;  // (rows: reverse looks at later tokens)
  int count;
  if (state) count = ntile;
  else count = rev ? ntile - tile : tile + 1;
  const int first = state ? (rev ? ntile - 1 : 0) : tile;
  const int dir = state ? (rev ? -1 : 1) : step;

  float4 nb[D / 16], nc[D / 16];
  const auto fetch_pair = [&](int n) {
    const int t0 = (first + n * dir) * C;
    fetch_tile<TIn, D>(nb, b + (size_t)t0 * sT, sT, L - t0, tid);
    fetch_tile<TIn, D>(nc, c + (size_t)t0 * sT, sT, L - t0, tid);
  };
  if (grp < count) fetch_pair(grp);
  if (!state && grp == G - 1) {
    float4 na[D / 16];
    const TIn* a = static_cast<const TIn*>(args.a) + head_off;
    fetch_tile<TIn, D>(na, a + (size_t)tile * C * sT, sT, L - tile * C, tid);
    put_tile<D, D + 4>(sm.a, na, tid);
  }
  for (int n = threadIdx.x; n <= L; n += ROWS_THREADS * G) sm.dtab[n] = decay_pow_d(s2, (double)n);
  __syncthreads();

  // The tiles of the entry state, after the others: one group at d = 128 takes them in a loop of their own (16 heads x 2048 tokens
  // forward 260 us in one loop, 253 this way; one group at d = 64 103.6 and 106.2).
  constexpr bool APART = D == 128 && G == 1;
  int items = count;
  if (!state) {
    // leave out the tiles whose every weight is zero in fp32, and add those of the entry state
    items = 1;
    while (items < count && sm.dtab[(items - 1) * C + 1] != 0.f) ++items;
    count = items;
    if (!APART && Z && sm.dtab[rev ? max(L - tile * C - C, 0) : tile * C + 1] != 0.f) items += D / C;
  }
  const auto fetch = [&](int n) {
    if (APART || n < count) fetch_pair(n);
    else fetch_tile<float, D>(nc, Z + (size_t)(n - count) * C * D, D, C, tid);
  };
  if (grp >= count && grp < items) fetch(grp);

  constexpr int EM = D / 16;  // value columns of a thread
  const int i4 = (tid / 16) * 4, e0 = (tid % 16) * 4;
  float acc[4][EM];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int m = 0; m < EM; ++m) acc[r][m] = 0.f;

  const auto accumulate = [&]() {
    // acc += w^T t over 32 rows; a thread has rows i4 .. i4 + 3 and columns e0 .. e0 + 3 (d = 128: and 64 + those)
#pragma unroll 4
    for (int j = 0; j < C; ++j) {
      const float4 w = *reinterpret_cast<const float4*>(&gm.w[j][i4]);
      const float wr[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int g = 0; g < EM / 4; ++g) {
        const float4 t = *reinterpret_cast<const float4*>(&gm.t[j][e0 + 64 * g]);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          acc[r][4 * g + 0] = fmaf(wr[r], t.x, acc[r][4 * g + 0]);
          acc[r][4 * g + 1] = fmaf(wr[r], t.y, acc[r][4 * g + 1]);
          acc[r][4 * g + 2] = fmaf(wr[r], t.z, acc[r][4 * g + 2]);
          acc[r][4 * g + 3] = fmaf(wr[r], t.w, acc[r][4 * g + 3]);
        }
      }
    }
  };

  for (int n = grp; n < items; n += G) {
    const bool pair = APART || n < count;  // else 32 rows of the entry state
    const int jt = first + n * dir;
    if (pair) put_tile<D, D + 4>(gm.b, nb, tid);
    put_tile<D, D>(gm.t, nc, tid);
    group_sync<G>(grp);
    if (n + G < items) fetch(n + G);
    if (!pair) {
      const int k0 = (n - count) * C;
      for (int x = tid; x < C * C; x += ROWS_THREADS) {
        const int k = x / C, i = x % C;
        const int dist = rev ? L - 1 - (tile * C + i) : tile * C + i + 1;
        gm.w[k][i] = dist >= 0 && dist <= L ? sm.a[i][k0 + k] * sm.dtab[dist] : 0.f;
      }
    } else if (state) {
      for (int x = tid; x < C * C; x += ROWS_THREADS) {
        const int j = x / C, i = x % C, t = jt * C + j;
        gm.w[j][i] = t < L ? gm.b[j][tile * C + i] * sm.dtab[rev ? t + 1 : L - 1 - t] : 0.f;
      }
    } else {
      // scores: a thread has rows i2, i2 + 1 and columns jc + 8 x
      const int i2 = (tid / 8) * 2, jc = tid % 8;
      float s[2][4];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int x = 0; x < 4; ++x) s[r][x] = 0.f;
#pragma unroll 4
      for (int k = 0; k < D; k += 4) {
        float4 av[2], bv[4];
#pragma unroll
        for (int r = 0; r < 2; ++r) av[r] = *reinterpret_cast<const float4*>(&sm.a[i2 + r][k]);
#pragma unroll
        for (int x = 0; x < 4; ++x) bv[x] = *reinterpret_cast<const float4*>(&gm.b[jc + 8 * x][k]);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            s[r][x] = fmaf(av[r].x, bv[x].x, s[r][x]);
            s[r][x] = fmaf(av[r].y, bv[x].y, s[r][x]);
            s[r][x] = fmaf(av[r].z, bv[x].z, s[r][x]);
            s[r][x] = fmaf(av[r].w, bv[x].w, s[r][x]);
          }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int i = i2 + r, j = jc + 8 * x;
          const int dist = rev ? (jt - tile) * C + j - i : (tile - jt) * C + i - j;
          // a select, not a multiply by zero: masked-out tokens can never leak
          gm.w[j][i] = dist >= 0 && jt * C + j < L ? s[r][x] * sm.dtab[min(dist, L)] : 0.f;
        }
    }
    group_sync<G>(grp);
    accumulate();
    group_sync<G>(grp);
  }
  if (APART && !state && Z && sm.dtab[rev ? max(L - tile * C - C, 0) : tile * C + 1] != 0.f) {
    for (int k0 = 0; k0 < D; k0 += C) {
      fetch_tile<float, D>(nc, Z + (size_t)k0 * D, D, C, tid);
      put_tile<D, D>(gm.t, nc, tid);
      for (int x = tid; x < C * C; x += ROWS_THREADS) {
        const int k = x / C, i = x % C;
        const int dist = rev ? L - 1 - (tile * C + i) : tile * C + i + 1;
        gm.w[k][i] = dist >= 0 && dist <= L ? sm.a[i][k0 + k] * sm.dtab[dist] : 0.f;
      }
      __syncthreads();
      accumulate();
      __syncthreads();
    }
  }
  if (G > 1) {
    // the groups' sums, in order, through their own tiles
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int g = 0; g < EM / 4; ++g)
        if (grp > 0)
          *reinterpret_cast<float4*>(&gm.t[i4 + r][e0 + 64 * g]) = make_float4(acc[r][4 * g], acc[r][4 * g + 1], acc[r][4 * g + 2], acc[r][4 * g + 3]);
    __syncthreads();
    if (grp > 0) return;
    for (int x = 1; x < G && x < items; ++x)
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int g = 0; g < EM / 4; ++g) {
          const float4 v = *reinterpret_cast<const float4*>(&sm.group[x].t[i4 + r][e0 + 64 * g]);
          acc[r][4 * g + 0] += v.x; acc[r][4 * g + 1] += v.y; acc[r][4 * g + 2] += v.z; acc[r][4 * g + 3] += v.w;
        }
  }

  if (state) {
    // state leaving the last segment: lambda^L Z + sum
    const bool local = args.local_out != nullptr;
    float* dst = (local ? args.local_out + ((size_t)bh * args.nseg + seg) * D * D : args.final_out + (size_t)bh * D * D) + (size_t)tile * C * D;
    const float gam = sm.dtab[L];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int gq = 0; gq < EM / 4; ++gq) {
        const size_t at = (size_t)(i4 + r) * D + e0 + 64 * gq;
        float4 z = Z ? *reinterpret_cast<const float4*>(Z + (size_t)tile * C * D + at) : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(dst + at) = make_float4(fmaf(gam, z.x, acc[r][4 * gq]), fmaf(gam, z.y, acc[r][4 * gq + 1]),
                                                           fmaf(gam, z.z, acc[r][4 * gq + 2]), fmaf(gam, z.w, acc[r][4 * gq + 3]));
      }
    return;
  }
  TOut* out = static_cast<TOut*>(args.out) + head_off;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = tile * C + i4 + r;
    if (i >= L) continue;
#pragma unroll
    for (int g = 0; g < EM / 4; ++g) {
      const float v[4] = {acc[r][4 * g], acc[r][4 * g + 1], acc[r][4 * g + 2], acc[r][4 * g + 3]};
      Vec4<TOut>::store(out + (size_t)i * sT + e0 + 64 * g, v);
    }
  }
}

// Whether a launch's tiles are shared out over groups.  With groups one thread block has a multiprocessor to itself (its registers),
// with one group four run at d = 64 and three at d = 128, but each ends sooner: the more tiles its rows add up, the more thread blocks a
// launch may have.  Measured, us, one group and four at d = 64: 37 heads x 512 (592 thread blocks, 16 tiles) 59 and 36, 64 x 512 (1024)
// 63 and 58, 75 x 512 (1200) 66 and 69, 90 x 200 (630, 7 tiles) 32.5 and 30.8, 90 x 300 (900, 10 tiles) 43 and 47, 140 x 128 (560, 4
// tiles) 22.5 and 24.3, 200 x 64 (400, 2 tiles) 12.4 and 15.9; one (two thread blocks to a multiprocessor, see rows_two_at_a_time) and
// two at d = 128: 19 x 500 (304) 70 and 50, 55 x 512 (880) 90 and 81, 64 x 512 (1024) 88 and 95, 50 x 300 (500, 10 tiles) 54 and 42, 70 x
// 300 (700) 56 and 58, 90 x 300 (900) 65 and 72, 60 x 200 (420, 7 tiles) 37 and 33, 90 x 200 (630) 43 and 47, 70 x 160 (350, 5 tiles) 29 and
// 26, 100 x 150 (500) 33 and 36; a backward pass's three walks at d = 128: 19 x 500 (912) 111 and 100, 30 x 300 (900) 84 and 76, 70 x 160
// (1050, 5 tiles) 64 and 70.  Short segments of a longer sequence, and states: 592 and 296.
inline bool rows_shared(int d, const RowsArgs& ra) {
  const int blocks = ra.first_block[ROWS_MAX_JOBS], tiles = ra.units[0] ? (ra.job[0].seg_len + C - 1) / C : 0;
  if (tiles >= 5 && d == 64) return blocks <= 300 + 55 * tiles;
  if (tiles >= 5) return blocks <= (ra.units[1] ? 550 + 40 * tiles : 200 + 44 * tiles);
  if (d == 64 && tiles > 0 && ra.job[0].nseg == 1) return blocks <= (tiles == 4 ? 444 : 296);
  return blocks <= (d == 64 ? 592 : 296);
}
// d = 128, one group, one walk of one segment: where a multiprocessor has two or three thread blocks' worth of rows, two at a time end
// before three do, whose longest rows wait for one another.  us, three and two: 100 heads x 128 (400 thread blocks, 4 tiles) 31 and 27, 125 x
// 128 (500) 33 and 28, 140 x 128 (560) 31 and 33, 75 x 512 (1200, 16 tiles) 108 and 99, 100 x 300 (1000, 10 tiles) 72 and 72, 100 x 400
// (1300, 13 tiles) 94 and 101, 200 x 160 (1000, 5 tiles) 53 and 59.
inline bool rows_two_at_a_time(const RowsArgs& ra) {
  if (!ra.units[0] || ra.units[1] || ra.job[0].nseg > 1) return false;
  const int blocks = ra.first_block[ROWS_MAX_JOBS], tiles = (ra.job[0].seg_len + C - 1) / C;
  return tiles >= 5 ? blocks <= 400 + 55 * tiles : blocks < 140 * tiles;
}
template <typename TIn, typename TOut, int D, int G>
cudaError_t launch_rows_g(const RowsArgs& ra, const DecayTable& tab, cudaStream_t stream) {
  constexpr size_t OWN = sizeof(RowsSmem<D, G>), TWO = 80 * 1024;  // (of TWO a multiprocessor has no room for three)
  constexpr bool CHOICE = D == 128 && G == 1;
  const size_t smem = CHOICE && rows_two_at_a_time(ra) ? TWO : OWN;
  auto kern = simt_rows_kernel<TIn, TOut, D, G>;
  // (the same limit from every thread that launches)
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(CHOICE ? TWO : OWN));
  if (err != cudaSuccess) return err;
  KernelTimer timer(ra.units[0] ? K_WALK : K_PREPASS, stream);
  // One walk of one segment by one group, all thread blocks at once: placed while the launch before still drains, long tiles come to
  // share multiprocessors (d = 64, 250 heads x 64 tokens 20.3 us, launched after it 14.4; d = 128, 100 x 128 35.8 and 30.9; the three
  // walks of a backward pass, d = 128, 74 x 64, 20.0 and 21.1).
  const bool early = G > 1 || !ra.units[0] || ra.units[1] || ra.job[0].nseg > 1 || ra.first_block[ROWS_MAX_JOBS] > 148 * (D == 64 ? 4 : 3);
  err = launch_kernel(early, kern, dim3((unsigned)ra.first_block[ROWS_MAX_JOBS]), dim3(ROWS_THREADS * G), smem, stream, 1, ra, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}
template <typename TIn, typename TOut, int D>
cudaError_t launch_rows_t(const RowsArgs& ra, const DecayTable& tab, cudaStream_t stream) {
  constexpr int MANY = D == 64 ? 4 : 2;
  return rows_shared(D, ra) ? launch_rows_g<TIn, TOut, D, MANY>(ra, tab, stream) : launch_rows_g<TIn, TOut, D, 1>(ra, tab, stream);
}
template <int D>
cudaError_t launch_rows_dims(const RowsArgs& ra, const DecayTable& tab, int in_dt, int out_dt, cudaStream_t stream) {
  if (in_dt == DT_F32 && out_dt == DT_F32) return launch_rows_t<float, float, D>(ra, tab, stream);
  if (in_dt == DT_BF16 && out_dt == DT_F32) return launch_rows_t<__nv_bfloat16, float, D>(ra, tab, stream);
  if (in_dt == DT_BF16 && out_dt == DT_BF16) return launch_rows_t<__nv_bfloat16, __nv_bfloat16, D>(ra, tab, stream);
  return cudaErrorInvalidValue;
}

template <typename TIn, typename TOut, int DA, int EC>
cudaError_t launch_walk_t(const OpArgs& args, const DecayTable& tab, cudaStream_t stream) {
  const size_t smem = sizeof(Smem<DA, EC>);
  const dim3 grid((unsigned)(args.BH * args.nseg)), block(THREADS);
  cudaError_t err;
  KernelTimer timer(K_WALK, stream);
  if (args.reverse) {
    auto kern = simt_walk_kernel<TIn, TOut, DA, EC, true>;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<grid, block, smem, stream>>>(args, tab);
  } else {
    auto kern = simt_walk_kernel<TIn, TOut, DA, EC, false>;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<grid, block, smem, stream>>>(args, tab);
  }
  count_launch();
  return cudaGetLastError();
}

template <typename TIn, int DA, int EC>
cudaError_t launch_prepass_t(const OpArgs& args, const DecayTable& tab, cudaStream_t stream) {
  const size_t smem = sizeof(PreSmem<TIn, DA, EC>);
  const dim3 grid((unsigned)(args.BH * args.nseg)), block(THREADS);
  cudaError_t err;
  KernelTimer timer(K_PREPASS, stream);
  if (args.reverse) {
    auto kern = simt_prepass_kernel<TIn, DA, EC, true>;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<grid, block, smem, stream>>>(args, tab);
  } else {
    auto kern = simt_prepass_kernel<TIn, DA, EC, false>;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<grid, block, smem, stream>>>(args, tab);
  }
  count_launch();
  return cudaGetLastError();
}

template <int DA, int EC>
cudaError_t launch_walk_dims(const OpArgs& args, const DecayTable& tab, int in_dt, int out_dt,
                             cudaStream_t stream) {
  if (in_dt == DT_F32 && out_dt == DT_F32) return launch_walk_t<float, float, DA, EC>(args, tab, stream);
  if (in_dt == DT_BF16 && out_dt == DT_F32)
    return launch_walk_t<__nv_bfloat16, float, DA, EC>(args, tab, stream);
  if (in_dt == DT_BF16 && out_dt == DT_BF16)
    return launch_walk_t<__nv_bfloat16, __nv_bfloat16, DA, EC>(args, tab, stream);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_simt_walk(const OpArgs& args, const DecayTable& tab, int Da, int Ec, int in_dt,
                             int out_dt, cudaStream_t stream) {
  if (Da == 64 && Ec == 64) return launch_walk_dims<64, 64>(args, tab, in_dt, out_dt, stream);
  if (Da == 128 && Ec == 128) return launch_walk_dims<128, 128>(args, tab, in_dt, out_dt, stream);
  return cudaErrorInvalidValue;
}

// Up to three independent walks, or the local states of one (local_out), in one launch; segments of at most ROWS_MAX_SEG tokens.
cudaError_t launch_simt_rows(const OpArgs* jobs, int njobs, const DecayTable& tab, int D, int in_dt, int out_dt,
                             cudaStream_t stream) {
  if (njobs < 1 || njobs > ROWS_MAX_JOBS || (D != 64 && D != 128)) return cudaErrorInvalidValue;
  RowsArgs ra{};
  long at = 0;
  for (int j = 0; j < ROWS_MAX_JOBS; ++j) {
    ra.first_block[j] = (int)at;
    if (j >= njobs) continue;
    const OpArgs& a = jobs[j];
    if (a.seg_len > ROWS_MAX_SEG) return cudaErrorInvalidValue;
    const long tiles = (std::min(a.seg_len, a.N) + C - 1) / C;
    const long rows = a.local_out ? 0 : (long)a.BH * a.nseg * tiles;
    const long states = a.local_out ? (long)a.BH * a.nseg * (D / C) : a.final_out ? (long)a.BH * (D / C) : 0;
    ra.job[j] = a;
    ra.job[j].seg_len = (int)std::min((long)a.seg_len, tiles * C);
    ra.units[j] = (int)rows;
    at += rows + states;
    if (at > 2147483647L) return cudaErrorInvalidValue;
  }
  ra.first_block[ROWS_MAX_JOBS] = (int)at;
  return D == 64 ? launch_rows_dims<64>(ra, tab, in_dt, out_dt, stream) : launch_rows_dims<128>(ra, tab, in_dt, out_dt, stream);
}

cudaError_t launch_simt_prepass(const OpArgs& args, const DecayTable& tab, int Da, int Ec, int in_dt,
                                cudaStream_t stream) {
  if (args.seg_len <= ROWS_MAX_SEG) return launch_simt_rows(&args, 1, tab, Da, in_dt, DT_F32, stream);
  if (Da == 64 && Ec == 64) {
    return in_dt == DT_F32 ? launch_prepass_t<float, 64, 64>(args, tab, stream)
                           : launch_prepass_t<__nv_bfloat16, 64, 64>(args, tab, stream);
  }
  if (Da == 128 && Ec == 128) {
    return in_dt == DT_F32 ? launch_prepass_t<float, 128, 128>(args, tab, stream)
                           : launch_prepass_t<__nv_bfloat16, 128, 128>(args, tab, stream);
  }
  return cudaErrorInvalidValue;
}

// One thread per four consecutive state elements; the pieces are few (ranks of a sequence-parallel group, or the
// segments of one chunk), so the sequential chain is short and every access is a coalesced 16-byte one.
__global__ void __launch_bounds__(256) chain_kernel(const ChainArgs args, const DecayTable tab) {
  // Every piece but the sequence's last is whole: two powers, formed once per thread block, which lies in one state.  (In
  // double by every thread and for every piece they took longer than the sums: 65536 tokens, 32 heads, 32 segments of
  // 2048 tokens 107 us with the states, 97 this way; 64 segments 182 and 164.)
  __shared__ float power[2];
  grid_dep_wait();
  grid_dep_launch();
  const long per_head = args.DE / 4;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int bh = (int)(i / per_head);
  const size_t e0 = (size_t)(i % per_head) * 4;
  const long long last = (args.N + args.piece_len - 1) / args.piece_len - 1;
  if (threadIdx.x < 2)
    power[threadIdx.x] = decay_pow_d(tab.s2[bh % args.H], (double)(threadIdx.x ? args.N - last * args.piece_len : args.piece_len));
  float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  if (args.z_in) z = *reinterpret_cast<const float4*>(args.z_in + (size_t)bh * args.DE + e0);
  const float* src = args.src + (size_t)bh * args.stride_bh + e0;
  __syncthreads();
  const float g_whole = power[0], g_last = power[1];
  int j = args.first;
#pragma unroll 4
  for (int n = 0; n < args.count; ++n, j += args.step) {
    const float g = j == last ? g_last : g_whole;
    const float4 x = *reinterpret_cast<const float4*>(src + (size_t)j * args.stride_j);
    z.x = fmaf(g, z.x, x.x);
    z.y = fmaf(g, z.y, x.y);
    z.z = fmaf(g, z.z, x.z);
    z.w = fmaf(g, z.w, x.w);
  }
  *reinterpret_cast<float4*>(args.out + (size_t)bh * args.DE + e0) = z;
}

cudaError_t launch_chain(const ChainArgs& args, const DecayTable& tab, cudaStream_t stream) {
  if (args.DE % 1024 != 0 || args.BH < 1 || args.count < 0 || args.piece_len < 1) return cudaErrorInvalidValue;
  const long threads = (long)args.BH * (args.DE / 4);
  KernelTimer timer(K_SCAN, stream);
  const cudaError_t err = launch_early(chain_kernel, dim3((unsigned)(threads / 256)), dim3(256), 0, stream, 1, args, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

// One thread per four state elements; the next segment's state is fetched one step ahead.
__global__ void __launch_bounds__(256) prefix_kernel(const ScanArgs args, const DecayTable tab) {
  grid_dep_wait();
  grid_dep_launch();
  const int bh = blockIdx.y;
  const double s2 = tab.s2[bh % args.H];
  if (!slow_head((float)s2, args.seg_len)) return;
  const int n_tok = args.seq_len ? args.seq_len[bh / args.H] : args.N;
  const int nseg = (n_tok + args.seg_len - 1) / args.seg_len;
  if (nseg < 3) return;  // a single state is its own running sum
  const size_t DE = (size_t)args.Da * args.Ec;
  float4* buf = reinterpret_cast<float4*>(args.buf + (size_t)bh * args.nseg * DE) + blockIdx.x * 256 + threadIdx.x;
  const long step = (long)(DE / 4);
  const float full = decay_pow_d(s2, (double)args.seg_len);  // every segment but the sequence's last is whole
  // forward: segments 0 .. nseg - 2 (nothing reads the state after the last), reverse: nseg - 1 .. 1
  const long first = args.reverse ? nseg - 1 : 0, dir = args.reverse ? -1 : 1;
  float4 z = buf[first * step], next = buf[(first + dir) * step];
  for (int i = 1; i < nseg - 1; ++i) {
    const float4 x = next;
    if (i + 1 < nseg - 1) next = buf[(first + (i + 1) * dir) * step];
    z.x = fmaf(full, z.x, x.x);
    z.y = fmaf(full, z.y, x.y);
    z.z = fmaf(full, z.z, x.z);
    z.w = fmaf(full, z.w, x.w);
    buf[(first + i * dir) * step] = z;
  }
}

cudaError_t launch_prefix(const ScanArgs& args, const DecayTable& tab, cudaStream_t stream) {
  if ((args.Da * args.Ec) % 1024 != 0 || args.BH > 65535) return cudaErrorInvalidValue;
  KernelTimer timer(K_SCAN, stream);
  const cudaError_t err =
      launch_kernel(early_walks(args.BH, args.nseg, args.seg_len), prefix_kernel, dim3((unsigned)(args.Da * args.Ec / 1024), (unsigned)args.BH),
                    dim3(256), 0, stream, 1, args, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_scan(const ScanArgs& args, const DecayTable& tab, cudaStream_t stream) {
  if (args.nseg > SCAN_MAX_SEG || (args.Da % 32) != 0 || (args.Ec % 32) != 0) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)args.BH, (unsigned)((args.Da / 32) * (args.Ec / 32)));
  KernelTimer timer(K_SCAN, stream);
  const cudaError_t err = launch_early(scan_kernel, grid, dim3(256), 0, stream, 1, args, tab);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace la
