// LRPE-d (Eq. 1): the decayed score times a learnable rotation of the relative position,
//   a_ts = lambda^(t-s) sum_i q_t[i] k_s[i] cos(theta[h][i] (t - s)),   s <= t   (real part of the printed form).
// The rotation splits into one factor per position, cos(a - b) = cos a cos b + sin a sin b, so with the features
//   x_c[t] = x[t] cos(theta t),  x_s[t] = x[t] sin(theta t)       (t the absolute position)
// the score is q_c.k_c + q_s.k_s and the output is the sum of two runs of the decayed operator,
//   O = op(Q_c, K_c, V) + op(Q_s, K_s, V),
// each with its own d x e state (the state of the doubled feature dimension 2d, stored as [2,B,H,d,e]).
// This file holds the element-wise kernels around those two runs -- the feature map, the sum of the two
// results, the chain rule back through the feature map including the gradient of the angles -- and the
// entry points that sequence them with la_fwd / la_bwd on the caller's stream.
//
// Angles: theta t is formed in double and reduced to [-pi, pi] before the fp32 sincos, so positions far into a
// long context lose nothing to the size of the product.  The gradient of theta is a position-weighted sum,
//   dtheta_i = sum_t t (q_c gs - q_s gc)_i + the same for k,     gc, gs = gradients of the two feature halves,
// whose two parts cancel down to the relative-position result; per-tile partial sums are written out and
// added in a fixed order (double) by a second kernel, so the result is reproducible bit for bit.
#include <cstdint>
#include <initializer_list>

#include "../../include/la.h"
#include "la_common.cuh"

namespace la {
// Both halves of the features as one run over twice the batch (la_api.cu); the size is (size_t)-1 where that cannot be.
size_t halves_workspace(int op, const la_shape* half);
la_status halves_fwd(const la_shape* half, const void* q, const void* k, const void* v, const float* lambda_host, void* o, void* o2,
                     const float* kv_in, float* kv_out, void* workspace, size_t workspace_bytes, void* stream);
la_status halves_bwd(const la_shape* half, const void* q, const void* k, const void* v, const void* d_o, const float* lambda_host,
                     void* dq, void* dk, void* dv, void* dv2, const float* kv_in, const float* grad_kv_out, float* grad_kv_in,
                     void* workspace, size_t workspace_bytes, void* stream);
namespace {

constexpr int RUN = 16;  // consecutive tokens a group of d/4 lanes walks
// tokens of one (b,h) per block in the gradient kernel: 256 / (d/4) groups, 128 (d = 128) or 256 (d = 64)
__host__ __device__ constexpr int tile_tokens(int d) { return RUN * (1024 / d); }

__device__ __forceinline__ void rotation(float theta, long long pos, float* c, float* s) {
  double a = (double)theta * (double)pos;
  a -= 6.283185307179586476925 * rint(a * 0.159154943091895335769);
  sincosf((float)a, s, c);
}

struct Geometry {   // where token t of (b,h) lives: element offset b*sB + h*sH + t*sT (+ feature)
  long long sT, sH, sB;
  int B, H, N, d;
};

// The angles a call needs, once for all its kernels and batches: (cos, sin) of theta t at every RUN-th token, [H, runs, d],
// and of theta itself behind them, [H, d].  The kernels get the tokens between by rotating (cos, sin) by the feature's own
// step angle, four multiply-adds instead of a sincos per element; over 16 steps the recurrence
// drifts by a few 1e-7, far below the bf16 features' 2^-9.  With the double products and sincos in the kernels themselves
// a warp spent most of its 2100 instructions on them with nothing in flight (this kernel: 7 us at 16 heads x 8192 tokens).
__global__ void __launch_bounds__(256) lrpe_angle_kernel(const float* theta, float2* table, int H, int d,
                                                         int runs, long long pos0) {
  grid_dep_wait();
  grid_dep_launch();
  const int hd = H * d, chunks = (hd + 255) / 256;
  const int run = blockIdx.x / chunks, i = blockIdx.x % chunks * 256 + threadIdx.x;  // run == runs: the step angles
  if (i >= hd) return;
  float2 v;
  rotation(theta[i], run < runs ? pos0 + (long long)run * RUN : 1, &v.x, &v.y);
  table[run < runs ? ((size_t)(i / d) * runs + run) * d + i % d : (size_t)runs * hd + i] = v;
}

// (cos, sin) of four consecutive features.
__device__ __forceinline__ void load_angles(const float2* at, float (&c)[4], float (&s)[4]) {
  const float4 x = *reinterpret_cast<const float4*>(at), y = *reinterpret_cast<const float4*>(at + 2);
  c[0] = x.x; s[0] = x.y; c[1] = x.z; s[1] = x.w;
  c[2] = y.x; s[2] = y.y; c[3] = y.z; s[3] = y.w;
}
__device__ __forceinline__ void turn(float (&c)[4], float (&s)[4], const float (&cs)[4], const float (&ss)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float cn = fmaf(c[k], cs[k], -s[k] * ss[k]);
    s[k] = fmaf(s[k], cs[k], c[k] * ss[k]);
    c[k] = cn;
  }
}

// x -> x cos(theta t), x sin(theta t) for x = q and k, same layout as x.  d/4 lanes share a token (four features each) and
// walk a run of RUN consecutive tokens of one (b,h).  Bound by memory, 12 bytes a feature of q and k in bf16; BATCH tokens of
// both are loaded before any is used (1 x 16 x 8192 x 128: 33 us, one tensor a launch
// and a sincos in the kernel 66).
constexpr int BATCH = 4;

template <typename T>
struct FeatureArgs {
  const T* x[2];  // q, k
  T* c[2];
  T* s[2];
};

template <typename T>
__device__ __forceinline__ void store_features(const FeatureArgs<T>& io, size_t off, const float (&q)[4], const float (&k)[4],
                                               const float (&c)[4], const float (&s)[4]) {
  const float qc[4] = {q[0] * c[0], q[1] * c[1], q[2] * c[2], q[3] * c[3]}, qs[4] = {q[0] * s[0], q[1] * s[1], q[2] * s[2], q[3] * s[3]};
  const float kc[4] = {k[0] * c[0], k[1] * c[1], k[2] * c[2], k[3] * c[3]}, ks[4] = {k[0] * s[0], k[1] * s[1], k[2] * s[2], k[3] * s[3]};
  Vec4<T>::store(io.c[0] + off, qc);
  Vec4<T>::store(io.s[0] + off, qs);
  Vec4<T>::store(io.c[1] + off, kc);
  Vec4<T>::store(io.s[1] + off, ks);
}

template <typename T>
__global__ void __launch_bounds__(256, 4) lrpe_feature_kernel(const FeatureArgs<T> io, const float2* table, Geometry g) {
  grid_dep_wait();
  grid_dep_launch();
  const int lanes = g.d >> 2;
  const int groups = 256 / lanes;
  const int lane = threadIdx.x % lanes, grp = threadIdx.x / lanes;
  const int c0 = lane * 4;
  const int runs_per_head = (g.N + RUN - 1) / RUN;
  const long total = (long)g.B * g.H * runs_per_head;
  for (long run = (long)blockIdx.x * groups + grp; run < total; run += (long)gridDim.x * groups) {
    const int t_first = (int)(run % runs_per_head) * RUN;
    const long bh = run / runs_per_head;
    const int h = (int)(bh % g.H), b = (int)(bh / g.H);
    float c[4], s[4], cs[4], ss[4];
    load_angles(table + ((size_t)h * runs_per_head + run % runs_per_head) * g.d + c0, c, s);
    load_angles(table + ((size_t)g.H * runs_per_head + h) * g.d + c0, cs, ss);
    size_t off = (size_t)b * g.sB + (size_t)h * g.sH + (size_t)t_first * g.sT + c0;
    int left = min(g.N - t_first, RUN);
    for (; left >= BATCH; left -= BATCH, off += BATCH * g.sT) {
      float v[2][BATCH][4];
#pragma unroll
      for (int n = 0; n < BATCH; ++n)
#pragma unroll
        for (int w = 0; w < 2; ++w) Vec4<T>::load(io.x[w] + off + n * g.sT, v[w][n]);
#pragma unroll
      for (int n = 0; n < BATCH; ++n) {
        store_features(io, off + n * g.sT, v[0][n], v[1][n], c, s);
        turn(c, s, cs, ss);
      }
    }
    for (; left > 0; --left, off += g.sT) {
      float v[2][4];
#pragma unroll
      for (int w = 0; w < 2; ++w) Vec4<T>::load(io.x[w] + off, v[w]);
      store_features(io, off, v[0], v[1], c, s);
      turn(c, s, cs, ss);
    }
  }
}

// dst = a + b (fp32 operands; dst may be a itself), four elements per thread.
template <typename TOut>
__global__ void __launch_bounds__(256) lrpe_sum_kernel(const float* a, const float* b, TOut* dst, long n4) {
  grid_dep_wait();
  grid_dep_launch();
  const long nthreads = (long)gridDim.x * blockDim.x;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += nthreads) {
    float x[4], y[4];
    Vec4<float>::load(a + 4 * i, x);
    Vec4<float>::load(b + 4 * i, y);
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] += y[k];
    Vec4<TOut>::store(dst + 4 * i, x);
  }
}

// Chain rule through the feature map, blockIdx.y = 0 for q and 1 for k:
//   dx = gc cos + gs sin,     part[(bh, tile), i] = sum over the tile's tokens of t (x cos gs - x sin gc)_i.
// Block = one tile of one (b,h); d/4 lanes share a token and walk a run of RUN.  Bound by memory (14
// bytes a feature): both in one launch, and the angles from the table (1 x 16 x 8192 x 128: 86 us,
// before 91; unrolled by two 98, its registers cost more warps than the loads ahead gain).

template <typename TIn, typename TOut>
struct GradArgs {
  const TIn* x[2];
  const float* gc[2];
  const float* gs[2];
  TOut* dx[2];
  float* part[2];
};

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(256) lrpe_grad_kernel(const GradArgs<TIn, TOut> io, const float2* table, Geometry g,
                                                           long long pos0, int ntiles) {
  __shared__ float red[2048];  // [tokens per pass][d]: 8 x 128 or 16 x 64
  grid_dep_wait();
  grid_dep_launch();
  const bool second = blockIdx.y != 0;
  const TIn* const x = second ? io.x[1] : io.x[0];
  const float* const gc = second ? io.gc[1] : io.gc[0];
  const float* const gs = second ? io.gs[1] : io.gs[0];
  TOut* const dx = second ? io.dx[1] : io.dx[0];
  float* const part = second ? io.part[1] : io.part[0];
  const int lanes = g.d >> 2;
  const int rows_per_pass = 256 / lanes;  // 8 (d = 128) or 16 (d = 64)
  const int lane = threadIdx.x % lanes, row0 = threadIdx.x / lanes;
  const int tile = blockIdx.x % ntiles, bh = blockIdx.x / ntiles;
  const int h = bh % g.H, b = bh / g.H;
  const int c0 = lane * 4;
  const size_t head_off = (size_t)b * g.sB + (size_t)h * g.sH + c0;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  const int t_first = tile * tile_tokens(g.d) + row0 * RUN;
  const int t_end = min(g.N, t_first + RUN);
  const int runs = (g.N + RUN - 1) / RUN;
  float c[4], s[4], cs[4], ss[4];
  load_angles(table + ((size_t)h * runs + min(t_first / RUN, runs - 1)) * g.d + c0, c, s);
  load_angles(table + ((size_t)g.H * runs + h) * g.d + c0, cs, ss);
  size_t off = head_off + (size_t)t_first * g.sT;
#pragma unroll 1
  for (int t = t_first; t < t_end; ++t, off += g.sT) {
    float v[4], a[4], bb[4], o[4];
    Vec4<TIn>::load(x + off, v);
    Vec4<float>::load(gc + off, a);
    Vec4<float>::load(gs + off, bb);
    const float pos = (float)(pos0 + t);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[k] = fmaf(a[k], c[k], bb[k] * s[k]);
      acc[k] = fmaf(pos, v[k] * (c[k] * bb[k] - s[k] * a[k]), acc[k]);
    }
    turn(c, s, cs, ss);
    Vec4<TOut>::store(dx + off, o);
  }
  // fixed-order sum over the token rows of the block
#pragma unroll
  for (int k = 0; k < 4; ++k) red[row0 * g.d + c0 + k] = acc[k];
  __syncthreads();
  if (threadIdx.x < g.d) {
    float s = 0.f;
    for (int r = 0; r < rows_per_pass; ++r) s += red[r * g.d + threadIdx.x];
    part[((size_t)bh * ntiles + tile) * g.d + threadIdx.x] = s;
  }
}

// dtheta[h][i] = sum over the batch and the tiles of the two partial arrays, in double, in an order that depends on
// the shape only (32 slices per feature: slice l adds the partials l, l + 32, ...; the slices are then added in
// order through shared memory), so the result is reproducible bit for bit.  Eight consecutive features per block.
__global__ void __launch_bounds__(256) lrpe_theta_reduce_kernel(const float* part_q,
                                                                const float* part_k,
                                                                float* dtheta, int B, int H, int ntiles, int d) {
  grid_dep_wait();
  grid_dep_launch();
  const int slice = threadIdx.x >> 3, fi = threadIdx.x & 7;
  const int idx = blockIdx.x * 8 + fi;  // feature index in [0, H*d)
  __shared__ double red[32][8];
  double s = 0.0;
  if (idx < H * d) {
    const int h = idx / d, i = idx % d;
    const int n = B * ntiles;
    for (int j = slice; j < n; j += 32) {
      const int b = j / ntiles, tl = j % ntiles;
      const size_t at = ((size_t)(b * H + h) * ntiles + tl) * d + i;
      s += (double)part_q[at] + (double)part_k[at];
    }
  }
  red[slice][fi] = s;
  __syncthreads();
  if (slice == 0 && idx < H * d) {
    double t = 0.0;
    for (int j = 0; j < 32; ++j) t += red[j][fi];
    dtheta[idx] = (float)t;
  }
}

unsigned grid_for(long threads_needed) {
  long blocks = (threads_needed + 255) / 256;
  const long cap = 148L * 16;
  return (unsigned)(blocks < 1 ? 1 : (blocks < cap ? blocks : cap));
}

Geometry geometry(const la_shape* s) {
  Geometry g;
  g.B = s->B; g.H = s->H; g.N = s->N; g.d = s->d;
  if (s->layout == LA_LAYOUT_BNHD) {
    g.sT = (long long)s->H * s->d; g.sH = s->d; g.sB = (long long)s->N * s->H * s->d;
  } else {
    g.sT = s->d; g.sH = (long long)s->N * s->d; g.sB = (long long)s->H * s->N * s->d;
  }
  return g;
}

size_t angle_count(const la_shape* s) { return (size_t)s->H * s->d * ((s->N + RUN - 1) / RUN + 1); }

cudaError_t run_angles(const la_shape* s, const float* theta, float2* table, long long pos0, cudaStream_t st) {
  KernelTimer timer(K_LRPE, st);
  const int runs = (s->N + RUN - 1) / RUN;
  const long blocks = (runs + 1L) * ((s->H * s->d + 255) / 256);
  if (blocks > 2147483647L) return cudaErrorInvalidValue;
  const cudaError_t err = launch_early(lrpe_angle_kernel, dim3((unsigned)blocks), dim3(256), 0, st, 1, theta, table, s->H, s->d, runs, pos0);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

template <typename T>
cudaError_t run_features_t(const la_shape* s, const void* q, const void* k, const float2* table, void* qc, void* qs, void* kc,
                           void* ks, cudaStream_t st) {
  KernelTimer timer(K_LRPE, st);
  FeatureArgs<T> io;
  io.x[0] = static_cast<const T*>(q); io.x[1] = static_cast<const T*>(k);
  io.c[0] = static_cast<T*>(qc); io.c[1] = static_cast<T*>(kc);
  io.s[0] = static_cast<T*>(qs); io.s[1] = static_cast<T*>(ks);
  const unsigned grid = grid_for((long)s->B * s->H * ((s->N + RUN - 1) / RUN) * (s->d / 4));
  const cudaError_t err = launch_early(lrpe_feature_kernel<T>, dim3(grid), dim3(256), 0, st, 1, io, table, geometry(s));
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}
cudaError_t run_features(const la_shape* s, const void* q, const void* k, const float2* table, void* qc, void* qs, void* kc,
                         void* ks, cudaStream_t st) {
  return s->in_dtype == LA_BF16 ? run_features_t<__nv_bfloat16>(s, q, k, table, qc, qs, kc, ks, st)
                                : run_features_t<float>(s, q, k, table, qc, qs, kc, ks, st);
}

cudaError_t run_sum(const la_shape* s, const float* a, const float* b, void* dst, cudaStream_t st) {
  KernelTimer timer(K_LRPE, st);
  const long n4 = (long)s->B * s->H * s->N * s->e / 4;
  const unsigned grid = grid_for(n4);
  const cudaError_t err =
      s->out_dtype == LA_BF16
          ? launch_early(lrpe_sum_kernel<__nv_bfloat16>, dim3(grid), dim3(256), 0, st, 1, a, b, (__nv_bfloat16*)dst, n4)
          : launch_early(lrpe_sum_kernel<float>, dim3(grid), dim3(256), 0, st, 1, a, b, (float*)dst, n4);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

// The tensors of GradArgs for q and k, untyped.
struct GradSet {
  const void* x;
  const float* gc;
  const float* gs;
  void* dx;
  float* part;
};
template <typename TIn, typename TOut>
cudaError_t run_grad_t(const la_shape* s, const GradSet& q, const GradSet& k, const float2* table, long long pos0, int ntiles,
                       cudaStream_t st) {
  KernelTimer timer(K_LRPE, st);
  GradArgs<TIn, TOut> io;
  for (int w = 0; w < 2; ++w) {
    const GradSet& one = w ? k : q;
    io.x[w] = static_cast<const TIn*>(one.x);
    io.gc[w] = one.gc;
    io.gs[w] = one.gs;
    io.dx[w] = static_cast<TOut*>(one.dx);
    io.part[w] = one.part;
  }
  const cudaError_t err = launch_early((lrpe_grad_kernel<TIn, TOut>), dim3((unsigned)((long)s->B * s->H * ntiles), 2), dim3(256), 0, st, 1, io, table, geometry(s), pos0, ntiles);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}
cudaError_t run_grad(const la_shape* s, const GradSet& q, const GradSet& k, const float2* table, long long pos0, int ntiles,
                     cudaStream_t st) {
  const bool ib = s->in_dtype == LA_BF16, ob = s->out_dtype == LA_BF16;
  if (ib && ob) return run_grad_t<__nv_bfloat16, __nv_bfloat16>(s, q, k, table, pos0, ntiles, st);
  if (ib) return run_grad_t<__nv_bfloat16, float>(s, q, k, table, pos0, ntiles, st);
  if (!ob) return run_grad_t<float, float>(s, q, k, table, pos0, ntiles, st);
  return cudaErrorInvalidValue;
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

// What la_fwd / la_bwd would reject, checked before the feature kernels are launched.
bool plain_args_ok(const la_shape* s, const float* lambda_host, std::initializer_list<const void*> ptrs) {
  if (!lambda_host) return false;
  for (int h = 0; h < s->H; ++h)
    if (!(lambda_host[h] > 0.f && lambda_host[h] <= 1.f)) return false;
  for (const void* p : ptrs)
    if (reinterpret_cast<uintptr_t>(p) & 15u) return false;
  return true;
}

// Workspace layout shared by the size query and the two entry points.
struct Carve {
  size_t feat;       // bytes of one feature tensor (in_dtype)
  size_t f32;        // bytes of one fp32 temporary of the tensors' size
  size_t part;       // bytes of one partial-sum array for dtheta
  size_t op;         // workspace of the inner la_fwd / la_bwd
  size_t angles;     // bytes of the angle table (forward: 0 where it lies in the temporary, which the runs write after the
                     // features are made)
  int ntiles;
  // One run over both halves: half the launches, and twice the heads to fill the chip with (1 x 16 heads x 8192, d = 128,
  // forward plus backward 660 us as two runs, 565 as one).  The halves of q and k and of their gradients lie one after the
  // other, so tensors may not be padded.
  bool one_run;
  int n_f32;         // fp32 temporaries
  size_t total;
};

bool carve(int op, const la_shape* s, Carve* c) {
  la_shape inner = *s;
  inner.out_dtype = LA_F32;
  size_t op_ws = la_workspace_bytes(op, &inner);
  if (op_ws == (size_t)-1 || s->d != s->e) return false;
  const size_t elems = (size_t)s->B * s->H * s->N * s->d;
  const size_t both = elems % 128 == 0 ? halves_workspace(op, &inner) : (size_t)-1;
  c->one_run = both != (size_t)-1;
  if (c->one_run) op_ws = both;
  c->feat = up256(elems * (s->in_dtype == LA_BF16 ? 2 : 4));
  c->f32 = up256(elems * 4);
  c->ntiles = (s->N + tile_tokens(s->d) - 1) / tile_tokens(s->d);
  c->part = up256((size_t)s->B * s->H * c->ntiles * s->d * 4);
  c->op = up256(op_ws);
  c->angles = up256(angle_count(s) * sizeof(float2));
  const bool out32 = s->out_dtype == LA_F32;
  if (op == LA_OP_FWD) {
    c->n_f32 = out32 ? 1 : 2;                    // the second half's result (and the first's when o is bf16)
    if (c->angles <= c->f32) c->angles = 0;
    c->total = 4 * c->feat + c->n_f32 * c->f32 + c->angles + c->op;
  } else {
    c->n_f32 = 4 + (out32 ? 1 : 2);              // gradients of the four feature tensors, dv of the halves
    c->total = 4 * c->feat + c->n_f32 * c->f32 + 2 * c->part + c->angles + c->op;
  }
  return true;
}

}  // namespace
}  // namespace la

using namespace la;

extern "C" {

size_t la_lrpe_workspace_bytes(int op, const la_shape* shape) {
  Carve c;
  if (!shape || (op != LA_OP_FWD && op != LA_OP_BWD) || !carve(op, shape, &c)) return (size_t)-1;
  return c.total;
}

la_status la_lrpe_fwd(const la_shape* shape, const void* q, const void* k, const void* v, const float* theta,
                      const float* lambda_host, long long pos0, void* o, const float* kv_in, float* kv_out,
                      void* workspace, size_t workspace_bytes, void* stream) {
  Carve c;
  if (!shape || !carve(LA_OP_FWD, shape, &c)) return shape ? LA_ERR_UNSUPPORTED : LA_ERR_INVALID_ARG;
  if (!q || !k || !v || !theta || !o || pos0 < 0) return LA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(theta) & 15u) || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return LA_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < c.total) return LA_ERR_WORKSPACE;
  if (!plain_args_ok(shape, lambda_host, {q, k, v, o, kv_in, kv_out})) return LA_ERR_INVALID_ARG;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(workspace);
  void* qc = w; void* qs = w + c.feat; void* kc = w + 2 * c.feat; void* ks = w + 3 * c.feat;
  float* tmp = reinterpret_cast<float*>(w + 4 * c.feat);
  float2* table = reinterpret_cast<float2*>(c.angles ? w + 4 * c.feat + c.n_f32 * c.f32 : w + 4 * c.feat);
  void* op_ws = w + 4 * c.feat + c.n_f32 * c.f32 + c.angles;
  const bool out32 = shape->out_dtype == LA_F32;
  la_shape inner = *shape;
  inner.out_dtype = LA_F32;
  const size_t state = (size_t)shape->B * shape->H * shape->d * shape->e;

  if (run_angles(shape, theta, table, pos0, cs) != cudaSuccess) return LA_ERR_CUDA;
  if (run_features(shape, q, k, table, qc, qs, kc, ks, cs) != cudaSuccess) return LA_ERR_CUDA;
  float* first = out32 ? static_cast<float*>(o) : tmp + c.f32 / 4;
  la_status st;
  if (c.one_run) {
    st = halves_fwd(&inner, qc, kc, v, lambda_host, first, tmp, kv_in, kv_out, op_ws, c.op, stream);
  } else {
    st = la_fwd(&inner, qc, kc, v, lambda_host, first, kv_in, kv_out, op_ws, c.op, stream);
    if (st == LA_OK)
      st = la_fwd(&inner, qs, ks, v, lambda_host, tmp, kv_in ? kv_in + state : nullptr, kv_out ? kv_out + state : nullptr,
                  op_ws, c.op, stream);
  }
  if (st != LA_OK) return st;
  if (run_sum(shape, first, tmp, o, cs) != cudaSuccess) return LA_ERR_CUDA;
  return LA_OK;
}

la_status la_lrpe_bwd(const la_shape* shape, const void* q, const void* k, const void* v, const void* d_o,
                      const float* theta, const float* lambda_host, long long pos0, void* dq, void* dk, void* dv,
                      float* d_theta, const float* kv_in, const float* grad_kv_out, float* grad_kv_in, void* workspace,
                      size_t workspace_bytes, void* stream) {
  Carve c;
  if (!shape || !carve(LA_OP_BWD, shape, &c)) return shape ? LA_ERR_UNSUPPORTED : LA_ERR_INVALID_ARG;
  if (!q || !k || !v || !d_o || !theta || !dq || !dk || !dv || !d_theta || pos0 < 0) return LA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(theta) & 15u) || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return LA_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < c.total) return LA_ERR_WORKSPACE;
  if (!plain_args_ok(shape, lambda_host, {q, k, v, d_o, dq, dk, dv, d_theta, kv_in, grad_kv_out, grad_kv_in}))
    return LA_ERR_INVALID_ARG;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(workspace);
  void* qc = w; void* qs = w + c.feat; void* kc = w + 2 * c.feat; void* ks = w + 3 * c.feat;
  w += 4 * c.feat;
  float* g_qc = reinterpret_cast<float*>(w);
  float* g_qs = reinterpret_cast<float*>(w + c.f32);
  float* g_kc = reinterpret_cast<float*>(w + 2 * c.f32);
  float* g_ks = reinterpret_cast<float*>(w + 3 * c.f32);
  float* dv_s = reinterpret_cast<float*>(w + 4 * c.f32);
  const bool out32 = shape->out_dtype == LA_F32;
  float* dv_c = out32 ? static_cast<float*>(dv) : reinterpret_cast<float*>(w + 5 * c.f32);
  w += c.n_f32 * c.f32;
  float* part_q = reinterpret_cast<float*>(w);
  float* part_k = reinterpret_cast<float*>(w + c.part);
  float2* table = reinterpret_cast<float2*>(w + 2 * c.part);
  void* op_ws = w + 2 * c.part + c.angles;
  la_shape inner = *shape;
  inner.out_dtype = LA_F32;
  const size_t state = (size_t)shape->B * shape->H * shape->d * shape->e;

  if (run_angles(shape, theta, table, pos0, cs) != cudaSuccess) return LA_ERR_CUDA;
  if (run_features(shape, q, k, table, qc, qs, kc, ks, cs) != cudaSuccess) return LA_ERR_CUDA;
  la_status st;
  if (c.one_run) {
    st = halves_bwd(&inner, qc, kc, v, d_o, lambda_host, g_qc, g_kc, dv_c, dv_s, kv_in, grad_kv_out, grad_kv_in, op_ws, c.op, stream);
    if (st != LA_OK) return st;
  } else {
    st = la_bwd(&inner, qc, kc, v, d_o, lambda_host, g_qc, g_kc, dv_c, kv_in, grad_kv_out, grad_kv_in, op_ws, c.op, stream);
    if (st != LA_OK) return st;
    st = la_bwd(&inner, qs, ks, v, d_o, lambda_host, g_qs, g_ks, dv_s, kv_in ? kv_in + state : nullptr,
                grad_kv_out ? grad_kv_out + state : nullptr, grad_kv_in ? grad_kv_in + state : nullptr, op_ws, c.op, stream);
    if (st != LA_OK) return st;
  }
  if (run_sum(shape, dv_c, dv_s, dv, cs) != cudaSuccess) return LA_ERR_CUDA;
  if (run_grad(shape, GradSet{q, g_qc, g_qs, dq, part_q}, GradSet{k, g_kc, g_ks, dk, part_k}, table, pos0, c.ntiles, cs) !=
      cudaSuccess)
    return LA_ERR_CUDA;
  {
    KernelTimer timer(K_LRPE, cs);
    const int n = shape->H * shape->d;
    const cudaError_t err = launch_early(lrpe_theta_reduce_kernel, dim3((unsigned)((n + 7) / 8)), dim3(256), 0, cs, 1, part_q, part_k, d_theta,
                                         shape->B, shape->H, c.ntiles, shape->d);
    count_launch();
    if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return LA_ERR_CUDA;
  }
  return LA_OK;
}

}  // extern "C"
