// Tensor-core kernels of the generic decayed linear-attention operator for bf16 inputs with Da = Ec = D, D = 128 or 64 (block
// formulas: la_common.cuh): the walks of la_tc_walk.cuh and la_tc_walk64.cuh, the segment states of la_tc_state.cuh, and what
// they share.  Operands that are formed on chip from fp32 values are carried as two bf16 terms hi + lo = x (to 2^-17), so that
// the only rounding left is the fp32 accumulation the method prescribes; each split can be turned off.
//
// Every group of warps that reads tensor memory has whole multiples of four warps, because a warp can only touch the 32-lane
// quarter given by its index mod 4.  All hand-offs are mbarriers; every wait is bounded and an expired wait makes the whole
// block unwind (flag set, copies drained, tensor memory freed).
//
// Shared-memory operand layouts are the canonical 128-byte-swizzled ones: K-major tiles as [128 rows][64 elements] panels (what
// a TMA box of 64 x 128 with CU_TENSOR_MAP_SWIZZLE_128B writes), MN-major tiles as [K rows][64 elements].
#include <cuda.h>

#include <cstddef>

#include "la_common.cuh"
#include "sm100_ptx.cuh"

namespace la {

__device__ unsigned int g_tc_status = 0;       // first non-zero failure code of any block (0 = none)
__device__ unsigned int g_tc_status_read = 0;  // where status_exchange_kernel leaves the value it took

namespace {
using namespace ptx;

constexpr int TMEM_COLS = 512;
constexpr long long WAIT_BUDGET = 2000000000LL;  // clocks (~1 s)

// One launch carries one job, or two jobs that walk the same tokens in the same direction (the dV and dK walks of
// the backward pass: they read the same four tensors, so the second read of each tile is an L2 hit).
struct TcJob {
  void* out;
  float* final_out;
  const float* z_in;  // the state entering the sequence and the segments' local states (see OpArgs)
  const float* local;
  bool z_in_t, local_t;
  int shared;  // see OpArgs
  // gate epilogue of the forward walk (D = 128 only): y = SRMSNorm(out) (.) u
  const void* u;
  void* y;
  float* rstd;
};

struct TcMaps {
  CUtensorMap a, b, c;
};

struct TcArgs {
  TcJob job[2];
  float* local_out;
  const int* seq_start;  // packed batch (see OpArgs): DEVICE arrays, or NULL
  const int* seq_len;
  const int* seq_order;
  int njobs;
  int BH, H, N, seg_len, nseg;
  int precision;
  int scanned, fold, follows;  // see OpArgs
  // D = 128: bytes to add to the first job's output for entries fold .. 2 fold - 1 (OpArgs::out2); D = 64: whether there is one
  long long second_half;
  long long sT, sH, sB;  // element offset of token t of (b,h): b*sB + h*sH + t*sT (rows of D contiguous features)
};

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                              long long budget = WAIT_BUDGET) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  // each try blocks in hardware for the default time limit (it returns early when the phase completes);
  // measured: giving a suspend-time hint of 1, 20 or 200 us instead makes the walk kernel 4 % slower
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > budget) return false;
  }
  return true;
}

// Used only while unwinding after a failure: waits (bounded) for work this thread started.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity) && clock64() - t0 < WAIT_BUDGET) {
  }
}

#define TC_WAIT_TO(label, barid, par, code)                              \
  do {                                                                   \
    if (!wait_or_abort(&sm.bars[barid], (par), &sm.abort)) {             \
      if (!sm.abort) atomicCAS(&g_tc_status, 0u, (unsigned)(code));      \
      sm.abort = 1;                                                      \
      goto label;                                                        \
    }                                                                    \
  } while (0)

// The same for a whole warp waiting together: the outcome is made warp-uniform so that the
// warp-level synchronisation of the elected arrivals below can never be entered by a part of a warp.
#define TC_WAIT_WARP_TO(label, barid, par, code)                                          \
  do {                                                                                    \
    const bool ok_ = wait_or_abort(&sm.bars[barid], (par), &sm.abort);                    \
    if (!__all_sync(0xffffffffu, ok_)) {                                                  \
      if (!ok_ && !sm.abort) atomicCAS(&g_tc_status, 0u, (unsigned)(code));               \
      sm.abort = 1;                                                                       \
      goto label;                                                                         \
    }                                                                                     \
  } while (0)
#define TC_WAIT_WARP(barid, par, code) TC_WAIT_WARP_TO(teardown, barid, par, code)

// One arrival per warp: every lane has fenced its own writes, the warp synchronises, lane 0
// arrives.  (A barrier that 256 threads arrive on costs 256 serialised shared-memory atomics per
// phase; at six such barriers per block that was a third of the kernel's shared-memory traffic.)
#define WARP_ARRIVE(barid)                               \
  do {                                                   \
    __syncwarp();                                        \
    if (lane == 0) mbar_arrive(&sm.bars[barid]);         \
  } while (0)

// Self-test of the failure path: one warp waits, with the kernels' own bounded wait, on a barrier that
// nothing ever arrives on; when the budget runs out it records code 99 like a real block would and returns.
__global__ void bounded_wait_selftest_kernel(long long budget) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (!wait_or_abort(&bar, 0, &abort_flag, budget)) {
    if (threadIdx.x == 0) atomicCAS(&g_tc_status, 0u, 99u);
  }
}

#include "la_tc_walk.cuh"
#include "la_tc_walk64.cuh"
#include "la_tc_state.cuh"

// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) return nullptr;
    if (q != cudaDriverEntryPointSuccess) return nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// Tensor map over a token tensor seen as {feature D, token N, head H, batch B} with element strides {1, sT, sH, sB}
// (D = 64 or 128, bf16 or fp32), a box of 128 bytes x box_tokens x 1 x 1 and 128-byte swizzle; tokens beyond N read
// as zero and are not written.  shared: one of the operands that the two halves of a folded batch have in common.
bool make_map(CUtensorMap* m, const void* ptr, const OpArgs& a, int D, bool f32 = false, int box_tokens = 128, bool shared = false) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  const cuuint64_t esz = f32 ? 4 : 2;
  // packed batch: one [total_tokens, H, D] tensor, batch extent 1
  const int B = a.seq_start ? 1 : shared ? a.fold : a.BH / a.H;
  const int tokens = a.seq_start ? a.total_tokens : a.N;
  cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)tokens, (cuuint64_t)a.H, (cuuint64_t)B};
  cuuint64_t strides[3] = {(cuuint64_t)a.sT * esz, (cuuint64_t)a.sH * esz, (cuuint64_t)a.sB * esz};
  cuuint32_t box[4] = {(cuuint32_t)(128 / esz), (cuuint32_t)box_tokens, 1, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return enc(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr),
             dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_maps(TcMaps* m, const OpArgs& args, int D) {
  return make_map(&m->a, args.a, args, D, false, 128, args.shared & SHARED_A) &&
         make_map(&m->b, args.b, args, D, false, 128, args.shared & SHARED_B) &&
         make_map(&m->c, args.c, args, D, false, 128, args.shared & SHARED_C);
}

TcJob make_job(const OpArgs& a) {
  return TcJob{a.out, a.final_out, a.z_in, a.local, a.z_in_t != 0, a.local_t != 0, a.shared, a.u, a.y, a.rstd};
}

TcArgs make_args(const OpArgs& args, const OpArgs* second, int precision) {
  TcArgs ta{};
  ta.job[0] = make_job(args);
  ta.job[1] = make_job(second ? *second : args);
  ta.local_out = args.local_out;
  ta.njobs = second ? 2 : 1;
  ta.BH = args.BH; ta.H = args.H; ta.N = args.N; ta.seg_len = args.seg_len; ta.nseg = args.nseg;
  ta.precision = precision;
  ta.scanned = args.scanned;
  ta.fold = args.fold;
  ta.follows = args.follows;
  ta.sT = args.sT; ta.sH = args.sH; ta.sB = args.sB;
  ta.seq_start = args.seq_start;
  ta.seq_len = args.seq_len;
  ta.seq_order = args.seq_order;
  return ta;
}

// One walk (second == nullptr) or two walks of the same direction over the same tokens in one launch.
cudaError_t launch_walk128(const OpArgs& args, const OpArgs* second, const DecayTable& tab, int out_dt, int precision,
                           cudaStream_t stream) {
  TcMaps m0, m1;
  if (!make_maps(&m0, args, 128)) return cudaErrorInvalidValue;
  m1 = m0;
  if (second && !make_maps(&m1, *second, 128)) return cudaErrorInvalidValue;
  const bool f32 = (out_dt == DT_F32);
  TcArgs ta = make_args(args, second, precision);
  if (second && second->out2) return cudaErrorInvalidValue;
  if (args.out2)
    ta.second_half = static_cast<char*>(args.out2) - static_cast<char*>(args.out) - args.fold * args.sB * (f32 ? 4 : 2);
  if (args.u) {  // the gate epilogue exists for the single forward walk
    if (second || args.reverse) return cudaErrorInvalidValue;
    if (args.out)
      return f32 ? launch_walk_t<false, float, 2>(m0, m1, ta, tab, stream)
                 : launch_walk_t<false, __nv_bfloat16, 2>(m0, m1, ta, tab, stream);
    return f32 ? launch_walk_t<false, float, 1>(m0, m1, ta, tab, stream)
               : launch_walk_t<false, __nv_bfloat16, 1>(m0, m1, ta, tab, stream);
  }
  if (args.reverse)
    return f32 ? launch_walk_t<true, float, 0>(m0, m1, ta, tab, stream)
               : launch_walk_t<true, __nv_bfloat16, 0>(m0, m1, ta, tab, stream);
  return f32 ? launch_walk_t<false, float, 0>(m0, m1, ta, tab, stream)
             : launch_walk_t<false, __nv_bfloat16, 0>(m0, m1, ta, tab, stream);
}

cudaError_t launch_walk64(const OpArgs& args, const OpArgs* second, const DecayTable& tab, int out_dt, int precision,
                          cudaStream_t stream) {
  const bool f32 = (out_dt == DT_F32);
  TcMaps m0, m1;
  VOutMaps out;
  if (args.u || (second && second->out2)) return cudaErrorInvalidValue;  // the gate: D = 128 only
  if (!make_maps(&m0, args, 64) || !make_map(&out.of[0], args.out, args, 64, f32, 128, args.out2 != nullptr)) return cudaErrorInvalidValue;
  m1 = m0;
  out.of[1] = out.second_half = out.of[0];
  if (second && (!make_maps(&m1, *second, 64) || !make_map(&out.of[1], second->out, *second, 64, f32))) return cudaErrorInvalidValue;
  if (args.out2 && !make_map(&out.second_half, args.out2, args, 64, f32, 128, true)) return cudaErrorInvalidValue;
  TcArgs ta = make_args(args, second, precision);
  ta.second_half = args.out2 != nullptr;
  if (args.reverse)
    return f32 ? launch_walk64_t<true, float>(m0, m1, out, ta, tab, stream)
               : launch_walk64_t<true, __nv_bfloat16>(m0, m1, out, ta, tab, stream);
  return f32 ? launch_walk64_t<false, float>(m0, m1, out, ta, tab, stream)
             : launch_walk64_t<false, __nv_bfloat16>(m0, m1, out, ta, tab, stream);
}

template <int D>
cudaError_t launch_states(const OpArgs& args, const DecayTable& tab, int precision, bool all_segments, cudaStream_t stream) {
  TcMaps m;
  if (!make_map(&m.b, args.b, args, D, false, 64, args.shared & SHARED_B) ||
      !make_map(&m.c, args.c, args, D, false, 64, args.shared & SHARED_C))
    return cudaErrorInvalidValue;
  const TcArgs ta = make_args(args, nullptr, precision);
  return args.reverse ? launch_state_t<true, D>(m, ta, tab, all_segments, stream)
                      : launch_state_t<false, D>(m, ta, tab, all_segments, stream);
}

}  // namespace

bool tc_supported() { return encode_fn() != nullptr; }

cudaError_t launch_tc_walk(const OpArgs& args, const DecayTable& tab, int D, int out_dt, int precision,
                           cudaStream_t stream) {
  return D == 128 ? launch_walk128(args, nullptr, tab, out_dt, precision, stream)
                  : launch_walk64(args, nullptr, tab, out_dt, precision, stream);
}

cudaError_t launch_tc_walk_pair(const OpArgs& first, const OpArgs& second, const DecayTable& tab, int D, int out_dt,
                                int precision, cudaStream_t stream) {
  if (first.reverse != second.reverse || first.N != second.N || first.BH != second.BH || first.nseg != second.nseg ||
      first.seg_len != second.seg_len)
    return cudaErrorInvalidValue;
  return D == 128 ? launch_walk128(first, &second, tab, out_dt, precision, stream)
                  : launch_walk64(first, &second, tab, out_dt, precision, stream);
}

cudaError_t launch_tc_prepass(const OpArgs& args, const DecayTable& tab, int D, int precision, bool all_segments,
                              cudaStream_t stream) {
  return D == 128 ? launch_states<128>(args, tab, precision, all_segments, stream)
                  : launch_states<64>(args, tab, precision, all_segments, stream);
}

cudaError_t launch_bounded_wait_selftest(long long budget_clocks, cudaStream_t stream) {
  bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>(budget_clocks);
  count_launch();
  return cudaGetLastError();
}

// Reads the failure flag and clears it in one atomic exchange on the device, so that a code recorded between
// a separate read and a separate clear cannot be lost.
__global__ void status_exchange_kernel(bool clear) {
  g_tc_status_read = clear ? atomicExch(&g_tc_status, 0u) : atomicAdd(&g_tc_status, 0u);
}

unsigned int tc_read_status(bool clear) {
  unsigned int v = 0;
  status_exchange_kernel<<<1, 1, 0, cudaStreamPerThread>>>(clear);
  if (cudaGetLastError() != cudaSuccess) return 0xFFFFFFFFu;
  if (cudaStreamSynchronize(cudaStreamPerThread) != cudaSuccess) return 0xFFFFFFFFu;
  if (cudaMemcpyFromSymbol(&v, g_tc_status_read, sizeof(v)) != cudaSuccess) return 0xFFFFFFFFu;
  return v;
}

}  // namespace la
