// Recurrent decode (iterations of Algorithm 2) for all (batch, head) pairs:
//   kv <- lambda kv + k v^T,   o <- kv^T q,   kv fp32 [BH, d, e] updated in place,
// for T >= 1 consecutive tokens per launch (q, k [BH, T, d], v, o [BH, T, e]): the state is read once, kept in
// registers over the T tokens and written once, so a few tokens decoded together (speculative or chunked
// decoding) cost one pass over the state instead of T.
//
// The step moves 2*d*e*4 bytes of state per (b,h) against 5*d*e flops, so it is
// bound by HBM bandwidth and runs on the plain fp32 ALUs.  One thread block owns
// one (b,h) state: every thread keeps a fixed group of four value columns and
// strides over the key rows, so a warp touches whole 512-byte rows with 16-byte
// accesses, all row loads are issued before the first use, and the column sums
// for o are reduced inside the block (no atomics, bitwise reproducible).
// With several tokens the inputs of up to CHUNK of them are fetched together with the state, so that a token costs its
// arithmetic and one barrier instead of a round trip to memory and two (16 x 32
// states, d = 128, 4 tokens: 14.8 us before, 13.5 now; 32 states, 8 tokens: 8.0 and 6.6).
#include "la_common.cuh"

namespace la {
namespace {

constexpr int THREADS = 256;
constexpr int CHUNK = 8;  // tokens whose inputs are on chip at a time

template <typename TIn, typename TOut, int D, int E>
__global__ void __launch_bounds__(THREADS)
decode_kernel(const TIn* q, const TIn* k, const TIn* v, float* kv, TOut* o, int H, int T, long long sT, long long sH, long long sB,
              const __grid_constant__ RateTable rates) {
  constexpr int LPR = E / 4;              // lanes per state row (float4 each)
  constexpr int RPP = THREADS / LPR;      // rows per pass
  constexpr int PASSES = D / RPP;
  static_assert(D == E && D % RPP == 0 && THREADS % LPR == 0, "shape");

  __shared__ alignas(16) float sq[CHUNK][D];  // (written, and sv read, 16 bytes at a time)
  __shared__ alignas(16) float sk[CHUNK][D];
  __shared__ alignas(16) float sv[CHUNK][E];
  __shared__ float4 red[2][RPP][LPR];

  grid_dep_wait();
  grid_dep_launch();
  const int bh = blockIdx.x;
  const int tid = threadIdx.x;
  const float lam = rates.lam[bh % H];
  const int col4 = tid % LPR;
  const int row0 = tid / LPR;

  float4* state = reinterpret_cast<float4*>(kv + (size_t)bh * D * E);
  const size_t head_off = (size_t)(bh / H) * sB + (size_t)(bh % H) * sH;  // token t of this (b,h): + t * sT

  // issue every state load first: PASSES independent 16-byte loads per thread
  float4 s[PASSES];
#pragma unroll
  for (int p = 0; p < PASSES; ++p) s[p] = ld_f4_streaming(&state[(size_t)(row0 + p * RPP) * LPR + col4]);

  for (int t = 0; t < T; ++t) {
    const int u = t % CHUNK;
    if (u == 0) {
      if (t > 0) __syncthreads();  // the chunk before has been read
      const int n = min(CHUNK, T - t);
      for (int x = tid; x < n * (D / 4); x += THREADS) {
        const size_t at = head_off + (size_t)(t + x / (D / 4)) * sT + x % (D / 4) * 4;
        float w[4];
        Vec4<TIn>::load(q + at, w);
        *reinterpret_cast<float4*>(&sq[x / (D / 4)][x % (D / 4) * 4]) = make_float4(w[0], w[1], w[2], w[3]);
        Vec4<TIn>::load(k + at, w);
        *reinterpret_cast<float4*>(&sk[x / (D / 4)][x % (D / 4) * 4]) = make_float4(w[0], w[1], w[2], w[3]);
        Vec4<TIn>::load(v + at, w);
        *reinterpret_cast<float4*>(&sv[x / (D / 4)][x % (D / 4) * 4]) = make_float4(w[0], w[1], w[2], w[3]);
      }
      __syncthreads();
    }
    const float4 vv = *reinterpret_cast<const float4*>(&sv[u][4 * col4]);

    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int p = 0; p < PASSES; ++p) {
      const int i = row0 + p * RPP;
      const float ki = sk[u][i], qi = sq[u][i];
      float4 x = s[p];
      x.x = fmaf(lam, x.x, ki * vv.x);
      x.y = fmaf(lam, x.y, ki * vv.y);
      x.z = fmaf(lam, x.z, ki * vv.z);
      x.w = fmaf(lam, x.w, ki * vv.w);
      s[p] = x;
      if (t == T - 1) __stcs(&state[(size_t)i * LPR + col4], x);  // the state leaves once, after the last token
      acc.x = fmaf(x.x, qi, acc.x);
      acc.y = fmaf(x.y, qi, acc.y);
      acc.z = fmaf(x.z, qi, acc.z);
      acc.w = fmaf(x.w, qi, acc.w);
    }
    red[t & 1][row0][col4] = acc;
    __syncthreads();
    if (tid < LPR) {
      float4 sum = red[t & 1][0][tid];
#pragma unroll
      for (int r = 1; r < RPP; ++r) {
        const float4 w = red[t & 1][r][tid];
        sum.x += w.x; sum.y += w.y; sum.z += w.z; sum.w += w.w;
      }
      TOut* op = o + head_off + (size_t)t * sT + 4 * tid;
      const float w[4] = {sum.x, sum.y, sum.z, sum.w};
      Vec4<TOut>::store(op, w);
    }
    // (red has two copies: the one read here is written again after the barrier of the next token)
  }
}

template <typename TIn, typename TOut, int D, int E>
cudaError_t launch_t(const void* q, const void* k, const void* v, float* kv, void* o, int BH, int H, int T,
                     long long sT, long long sH, long long sB, const RateTable& rates, cudaStream_t stream) {
  KernelTimer timer(K_DECODE, stream);
  const cudaError_t err = launch_early(decode_kernel<TIn, TOut, D, E>, dim3((unsigned)BH), dim3(THREADS), 0, stream, 1,
                                       static_cast<const TIn*>(q), static_cast<const TIn*>(k), static_cast<const TIn*>(v), kv,
                                       static_cast<TOut*>(o), H, T, sT, sH, sB, rates);
  count_launch();
  return err != cudaSuccess ? err : cudaGetLastError();
}

template <int D, int E>
cudaError_t launch_dims(const void* q, const void* k, const void* v, float* kv, void* o, int BH, int H, int T,
                        int in_dt, int out_dt, long long sT, long long sH, long long sB, const RateTable& rates,
                        cudaStream_t stream) {
  if (in_dt == DT_F32 && out_dt == DT_F32)
    return launch_t<float, float, D, E>(q, k, v, kv, o, BH, H, T, sT, sH, sB, rates, stream);
  if (in_dt == DT_BF16 && out_dt == DT_F32)
    return launch_t<__nv_bfloat16, float, D, E>(q, k, v, kv, o, BH, H, T, sT, sH, sB, rates, stream);
  if (in_dt == DT_BF16 && out_dt == DT_BF16)
    return launch_t<__nv_bfloat16, __nv_bfloat16, D, E>(q, k, v, kv, o, BH, H, T, sT, sH, sB, rates, stream);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_decode(const void* q, const void* k, const void* v, float* kv, void* o, int BH,
                          int H, int T, int d, int e, int in_dt, int out_dt, long long sT, long long sH, long long sB,
                          const RateTable& rates, cudaStream_t stream) {
  if (T < 1) return cudaErrorInvalidValue;
  if (d == 64 && e == 64) return launch_dims<64, 64>(q, k, v, kv, o, BH, H, T, in_dt, out_dt, sT, sH, sB, rates, stream);
  if (d == 128 && e == 128)
    return launch_dims<128, 128>(q, k, v, kv, o, BH, H, T, in_dt, out_dt, sT, sH, sB, rates, stream);
  return cudaErrorInvalidValue;
}

}  // namespace la
