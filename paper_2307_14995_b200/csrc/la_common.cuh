// Shared declarations of the CUDA side: kernel parameter blocks and the launch
// helpers that the C-ABI entry points in la_api.cu call.
//
// One generic operator covers forward and all three gradients.  With a
// "query-like" a [N,Da], a "key-like" b [N,Da] and a "value-like" c [N,Ec]:
//
//   forward direction   out_t = sum_{s<=t} lambda^(t-s) (a_t.b_s) c_s + lambda^(t+1)   Z_in^T a_t
//   reverse direction   out_t = sum_{s>=t} lambda^(s-t) (a_t.b_s) c_s + lambda^(N-1-t) Z_in^T a_t
//
// where Z is the Da x Ec running state sum_s decay * b_s c_s^T.  Then
//   O  = fwd(a=Q,  b=K,  c=V)        state = KV          (Algorithm 2 / Algorithm 3)
//   dQ = fwd(a=dO, b=V,  c=K)        state = KV^T        (Algorithm 4, dQ line)
//   dK = rev(a=V,  b=dO, c=Q)        state = (dKV)^T     (Algorithm 4, dK line)
//   dV = rev(a=K,  b=Q,  c=dO)       state = dKV         (Algorithm 4, dV line)
// The sequence is processed in blocks of C tokens (block-local index i, j):
//   out_blk = ((a b^T) (.) D) c + diag(f_out) a Z,      Z <- Gamma Z + b^T diag(f_state) c
// with every decay factor a non-negative power of lambda:
//   forward: D_ij = lambda^(i-j) [i>=j], f_out_i = lambda^(i+1),    f_state_j = lambda^(Cr-1-j)
//   reverse: D_ij = lambda^(j-i) [j>=i], f_out_i = lambda^(Cr-1-i), f_state_j = lambda^(j+1)
//   Gamma = lambda^Cr, Cr = number of real tokens in the block (a ragged last block
//   uses its own Cr so that no state is decayed through padding).
// Factors are evaluated as exp2(-s2 * n) with s2 = -log2(lambda) >= 0, never as a
// ratio of powers, so nothing can overflow and underflow only flushes to the
// correct limit 0 (this is what the prescaled form of Algorithm 1 cannot offer).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <utility>

#define LA_MAX_H 256

namespace la {

struct DecayTable {
  double s2[LA_MAX_H];  // -log2(lambda_h) >= 0, computed in double on the host
};

// Arguments of one generic-operator launch (either the walking kernel or the
// state-only pre-pass).
constexpr int SHARED_A = 1, SHARED_B = 2, SHARED_C = 4;
struct OpArgs {
  const void* a;      // [BH, N, Da]  (unused by the pre-pass)
  const void* b;      // [BH, N, Da]
  const void* c;      // [BH, N, Ec]
  void* out;          // [BH, N, Ec]  (unused by the pre-pass)
  const float* entry; // [BH, nseg, Da*Ec] state entering each segment, or NULL = zeros
  // Tensor-core walks instead of `entry`: the state entering the sequence [BH, Da*Ec] (NULL = zeros) and
  // the segments' local states [BH, nseg, Da*Ec] as the pre-pass leaves them, which the walk chains itself; each may be
  // stored transposed.
  const float* z_in;
  const float* local;
  int z_in_t, local_t;
  int scanned;  // launch_prefix has turned the local states of the slowly decaying heads into running ones
  float* local_out;   // pre-pass: [BH, nseg, Da*Ec] segment-local states
  float* final_out;   // [BH, Da*Ec] state leaving the last-processed segment, or NULL
  int BH, H, N;
  int seg_len, nseg;  // seg_len is a multiple of 128
  int reverse;        // 0 forward, 1 reverse
  int follows;        // tensor-core walk: Follows
  // Where token t of (batch b, head h) sits in a, b, c, out, u, y: element offset b*sB + h*sH + t*sT of a row of
  // Da / Ec contiguous features.  [B,H,N,D]: sT = D, sH = N*D, sB = H*N*D; [B,N,H,D]: sT = H*D, sH = D, sB = N*H*D
  // (D = Da = Ec in every supported shape).
  long long sT, sH, sB;
  // Optional epilogue of the forward walk (Eq. 3 with Eq. 8): y = SRMSNorm(out) (.) u per row.  With u set, y is
  // written, `out` becomes optional (NULL = the attention output itself is not wanted) and rstd [BH, N] optional.
  const void* u;      // [BH, N, Ec] gate, input dtype
  void* y;            // [BH, N, Ec] output dtype
  float* rstd;        // [BH, N] sqrt(Ec) / ||out row||_2, or NULL
  // Packed batch of sequences of different lengths (tensor-core kernels only; NULL elsewhere):
  // the token tensors are [total_tokens, H, D] with the sequences one after the other, "batch" entry b is
  // sequence b with seq_len[b] tokens starting at token seq_start[b] (DEVICE arrays of BH / H ints), N is the
  // longest length (it fixes the segment grid; thread blocks of segments a sequence does not have return at once)
  // and sB is unused.  Rows past a sequence's end belong to its neighbour, not to a zero-filled margin, so every
  // bound below is the sequence's own length.
  const int* seq_start;
  const int* seq_len;
  // Folded batch (tensor-core kernels only; 0 elsewhere): batch entries t and t + fold read the same
  // entry t of the operands in `shared` (SHARED_* bits), which have `fold` batch entries.
  // out2: where the entries fold .. 2 fold - 1 of the output go, as entries 0 .. fold - 1 (NULL: behind the others in `out`).
  int fold;
  int shared;
  void* out2;
  const int* seq_order;  // the order in which thread blocks take the sequences (longest first), or NULL
  int total_tokens;
};

struct ScanArgs {
  float* buf;          // [BH, nseg, Da*Ec]: in = segment-local states, out = entry states
  float* buf_t;        // optional transposed copy of the entry states [BH, nseg, Ec*Da]
  const float* z_in;   // [BH, Da*Ec] (or [BH, Ec*Da] if z_in_transposed), or NULL = zeros
  int z_in_transposed;
  int BH, H, N, seg_len, nseg, Da, Ec, reverse;
  const int* seq_len;  // launch_prefix, packed batch: DEVICE array of BH / H lengths (N is then the longest), or NULL
};

// Chain of piece-local states into the state at one boundary (a cut of the sequence):
//   forward (first <= last):  z = z_in;  for j = first .. last:      z = lambda^(L_j) z + src_j
//   reverse (first >  last):  z = z_in;  for j = first down to last: z = lambda^(L_j) z + src_j
// with L_j = tokens of piece j = min(N, (j+1) piece_len) - j piece_len.  count == 0 copies z_in (or zeros).
struct ChainArgs {
  const float* src;         // element i of piece j of (b,h): src[j * stride_j + bh * stride_bh + i]
  long long stride_j, stride_bh;
  const float* z_in;        // [BH, DE] or NULL = zeros
  float* out;               // [BH, DE]
  int BH, H, DE;
  int first, count, step;   // pieces first, first + step, ... (count of them), step = +1 or -1
  long long N, piece_len;
};

// dtype tags as in la.h
enum { DT_BF16 = 0, DT_F32 = 1 };

// Each returns cudaGetLastError() of its launch.
cudaError_t launch_simt_walk(const OpArgs& args, const DecayTable& tab, int Da, int Ec, int in_dt,
                             int out_dt, cudaStream_t stream);
// Up to three independent walks in one launch, with segments of at most ROWS_MAX_SEG tokens.
constexpr int ROWS_MAX_SEG = 512;
cudaError_t launch_simt_rows(const OpArgs* jobs, int njobs, const DecayTable& tab, int D, int in_dt, int out_dt,
                             cudaStream_t stream);
cudaError_t launch_simt_prepass(const OpArgs& args, const DecayTable& tab, int Da, int Ec, int in_dt,
                                cudaStream_t stream);
cudaError_t launch_scan(const ScanArgs& args, const DecayTable& tab, cudaStream_t stream);
// Running sums of the segments' local states, in place: afterwards buf[p] is the state leaving segment p with nothing
// entering the sequence.  Only for heads whose states reach over more than one segment (slow_head); args.buf, BH, H, N,
// seg_len, nseg, Da, Ec, reverse and seq_len are used.
cudaError_t launch_prefix(const ScanArgs& args, const DecayTable& tab, cudaStream_t stream);
// Whole segments of seg_len tokens through which a state can be followed before its decay is below 2^-160, exactly zero in
// fp32 (no limit for lambda = 1), and whether a head's states are worth a running sum.
__host__ __device__ inline float state_reach(float s2, int seg_len) { return s2 > 0.f ? 160.f / (s2 * (float)seg_len) : 3.0e38f; }
__host__ __device__ inline bool slow_head(float s2, int seg_len) { return state_reach(s2, seg_len) >= 2.f; }
cudaError_t launch_chain(const ChainArgs& args, const DecayTable& tab, cudaStream_t stream);
// The decay rates themselves, where a single power is all that is needed.
struct RateTable {
  float lam[LA_MAX_H];
};
// T >= 1 consecutive tokens per (batch, head); token t of (b,h) is the row at element offset b*sB + h*sH + t*sT.
cudaError_t launch_decode(const void* q, const void* k, const void* v, float* kv, void* o, int BH,
                          int H, int T, int d, int e, int in_dt, int out_dt, long long sT, long long sH, long long sB,
                          const RateTable& rates, cudaStream_t stream);

// SimpleRMSNorm followed by the gate as stand-alone row kernels (la_gate.cu): y = SRMSNorm(o) (.) u (o and y may be
// the same buffer), and the gradients of <y, dy> with respect to o (written in the input dtype) and u.
cudaError_t launch_norm_gate_fwd(const void* o, const void* u, void* y, float* rstd, long rows, int e, int in_dt,
                                 int out_dt, cudaStream_t stream);
cudaError_t launch_norm_gate_bwd(const void* o, const void* u, const void* dy, void* d_o, void* d_u, long rows, int e,
                                 int in_dt, int out_dt, cudaStream_t stream);

// Tensor-core (tcgen05) kernels: bf16 inputs, Da = Ec = D with D = 64 or 128.
bool tc_supported();
cudaError_t launch_tc_walk(const OpArgs& args, const DecayTable& tab, int D, int out_dt, int precision,
                           cudaStream_t stream);
// Two walks of the same direction over the same tokens (same N, BH, segments) in one launch; the thread blocks of
// the two are interleaved so that tiles both read come from HBM once.
cudaError_t launch_tc_walk_pair(const OpArgs& first, const OpArgs& second, const DecayTable& tab, int D, int out_dt,
                                int precision, cudaStream_t stream);
// all_segments: false leaves out the segment that no other segment's state depends on (forward the last, reverse the
// first).
cudaError_t launch_tc_prepass(const OpArgs& args, const DecayTable& tab, int D, int precision, bool all_segments,
                              cudaStream_t stream);

// One warp runs the kernels' bounded wait on a barrier nothing arrives on (budget in SM clocks).
cudaError_t launch_bounded_wait_selftest(long long budget_clocks, cudaStream_t stream);

// Failure code recorded by a tensor-core block whose bounded wait expired (0 = none);
// copies it from the device (blocking) and optionally clears it.
unsigned int tc_read_status(bool clear);

void count_launch(int n = 1);

// Launches that may begin while the launch before them on the stream ends (programmatic dependent launch).  A kernel lets its
// successor begin (grid_dep_launch) only after its own wait for its predecessor (grid_dep_wait), so whatever came before the
// predecessor is complete when a kernel begins; what the predecessor itself writes needs the wait.  Kernels that do not say
// otherwise (Follows) wait before their first access to memory.
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(bool early, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster,
                          Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2]{};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = early;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_early(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster, Args&&... args) {
  return launch_kernel(true, kern, grid, block, smem, stream, cluster, std::forward<Args>(args)...);
}
// Tensor-core walks and their states begin early where the thread blocks of one walk run all at once and are not long.  Where they
// come in several waves or run for long a launch's end matters less, and held at the power limit the step is slower for it: 1 x 32
// heads x 65536, 288 thread blocks a walk, 2333 us with launches one after the other and 2368 with early ones; 1 x 16 x 51521, 144
// thread blocks of 45 blocks, 920 and 932; 128 thread blocks: 1 x 32 x 16384, 32 blocks each, 639 and 634; 2 x 16 x 8192, 16 blocks,
// 333 and 320 (all on one box, in turn; runs of one side differ by half a percent).
inline bool early_walks(int bh, int nseg, int seg_len) { return (long)bh * nseg <= 148 && seg_len <= 4096; }
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// ... and loads come behind it: never through the read-only path (ld.global.nc: __ldg, or a const __restrict__ parameter of the kernel),
// which is for memory that nobody writes from a kernel's beginning on, nor by an instruction that the compiler may move ahead of the
// wait.  As instructions where it matters which registers they take: with C++ loads of its entry state the gated walk at d = 128 spills
// 48 bytes more (1 x 32 x 65536 in bf16 700 us, this way 660).
__device__ __forceinline__ float ld_f1(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_f4(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_f4_streaming(const float4* p) {  // evict-first
  float4 v;
  asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// What a walk needs of the launch before it on the stream.
// Tensor memory: a kernel takes its columns before it lets its successor begin, so a walk behind a launch of its own call (FOLLOWS_STATES,
// FOLLOWS_WALK) may take its own at once.  The first launch of a call waits first: what is ahead of it may be another library's kernel
// that let it begin with columns of its own still to come, which would then wait for a thread block that waits for it.
enum Follows {
  FOLLOWS_ANY = 0,     // the first launch of a call: everything
  FOLLOWS_STATES = 1,  // the states that it chains; its other inputs were complete before that launch began
  FOLLOWS_WALK = 2,    // nothing: a walk of the same call, which began when the states of both were complete
};

// Brackets one kernel launch with CUDA events when benchmark profiling is enabled
// (la_profile_enable); otherwise does nothing.  kind is one of LA_KERNEL_*.
struct KernelTimer {
  KernelTimer(int kind, cudaStream_t stream);
  ~KernelTimer();
  int kind_;
  cudaStream_t stream_;
  cudaEvent_t start_;
  bool active_;
};
enum { K_PREPASS = 0, K_SCAN = 1, K_WALK = 2, K_DECODE = 3, K_WALK_PAIR = 4, K_GATE = 5, K_LRPE = 6, K_NUM = 7 };

// ---- small device helpers --------------------------------------------------
__device__ __forceinline__ float decay_pow_d(double s2, double n) {
  // lambda^n for n >= 0 in double, rounded once; s2 == 0 (lambda == 1) gives exactly 1.
  return (float)exp2(-s2 * n);
}

// four consecutive elements as one vector access, widened to fp32
template <typename T> struct Vec4;
template <> struct Vec4<float> {
  static __device__ __forceinline__ void load(const float* p, float (&x)[4]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  }
  static __device__ __forceinline__ void store(float* p, const float (&x)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  }
};
template <> struct Vec4<__nv_bfloat16> {
  static __device__ __forceinline__ void load(const __nv_bfloat16* p, float (&x)[4]) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, const float (&x)[4]) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(x[0], x[1]), b = __floats2bfloat162_rn(x[2], x[3]);
    uint2 v;
    v.x = *reinterpret_cast<const uint32_t*>(&a);
    v.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = v;
  }
};

template <typename T> __device__ __forceinline__ float to_f32(T x);
template <> __device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) {
  return __bfloat162float(x);
}
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

}  // namespace la
