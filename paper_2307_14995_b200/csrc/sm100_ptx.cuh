// Inline-PTX wrappers for the Blackwell (sm_100a) features the tensor-core kernels
// use: mbarriers with bounded waits, TMA tiled loads/stores (no multicast), TMEM
// allocation, tcgen05.mma with shared-memory descriptors, tcgen05.ld.
//
// Every wait in this file gives up after a clock budget and reports failure to the
// caller, which records an error code and unwinds (frees TMEM, returns) instead of
// spinning forever.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace la {
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---- mbarrier ------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// ---- registers per thread of a warpgroup ----------------------------------------------------
template <int N>
__device__ __forceinline__ void reg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void reg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// This warp's registers per thread from now on, LAUNCH being what the launch gave: setmaxnreg.inc must not be given less
// than the warp has, nor .dec more (an illegal instruction).
template <int N, int LAUNCH>
__device__ __forceinline__ void set_regs() {
  if (N < LAUNCH) reg_dec<N>();
  if (N > LAUNCH) reg_inc<N>();
}

// ---- proxy / tcgen05 fences -------------------------------------------------------------------
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 2^x on the special-function unit (relative error 2^-22, denormal results flush to zero).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---- TMA (tiled, this CTA only; never multicast) ------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// The same for 4-D maps {feature, token, head, batch}.
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2),
      "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, const void* smem_src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(m)),
               "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until the smem sources of all committed bulk stores have been read.
__device__ __forceinline__ void tma_store_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}


// ---- TMEM ----------------------------------------------------------------------------------------
// One full warp allocates `ncols` (power of two >= 32) columns; the base address lands in *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot_smem)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ---- UMMA descriptors ------------------------------------------------------------------------------
// The same descriptor as two 32-bit halves.  Only the low half depends on the address, and a
// byte offset `off` (multiple of 16) inside one buffer moves it by off >> 4 (shared-memory
// addresses stay below 2^18, so the 14-bit field cannot carry).
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t smem_addr, uint32_t lbo_bytes) {
  return ((smem_addr & 0x3FFFFu) >> 4) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
constexpr uint32_t UMMA_DESC_HI_SBO1024 = (1024u >> 4) | (1u << 14) | (2u << 29);  // sbo = 1024, version, 128-byte swizzle

// Instruction descriptor for kind::f16 with bf16 A/B and fp32 accumulation.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N, bool a_mn_major, bool b_mn_major) {
  return (1u << 4)                       // D format: f32
         | (1u << 7)                     // A format: bf16
         | (1u << 10)                    // B format: bf16
         | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---- TMEM loads: 32 lanes x 32-bit, N consecutive columns per thread ------------------------------
__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, "
      "%25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// Sixteen lanes (those of taddr) x 64 columns: registers 4 x, 4 x + 1 of thread t are lane t / 4, columns 8 x + 2 (t % 4) and
// the next, registers 4 x + 2, 4 x + 3 the same columns of lane t / 4 + 8.
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, "
      "%25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- TMEM stores: 32 lanes x 32-bit, N consecutive columns per thread ---------------------------
__device__ __forceinline__ void tmem_st_x4(uint32_t taddr, const uint4& r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r.x), "r"(r.y), "r"(r.z),
               "r"(r.w)
               : "memory");
}
__device__ __forceinline__ void tmem_st_x16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// Sixteen lanes (those of taddr) x 8 columns: register 2 x of thread t is lane t / 4, column 4 x + t % 4, register
// 2 x + 1 lane t / 4 + 8 of the same column -- two by two 8 x 8 matrices of 16-bit pairs, each spread over the
// warp as ldmatrix leaves it.
__device__ __forceinline__ void tmem_st_16x128b_x2(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.16x128b.x2.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3])
               : "memory");
}
// The same with 32 columns.
__device__ __forceinline__ void tmem_st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// Four 8 x 8 matrices of 16-bit elements, transposed: thread t gets elements (row 2 (t % 4), row 2 (t % 4) + 1) of column
// t / 4 of each; lane 8 m + i supplies the address of row i of matrix m (16 bytes).
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t saddr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(saddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }


// ---- warp-convergent issue -------------------------------------------------------------------------
// The MMA-issuing warp runs its whole loop with all 32 lanes converged and
// only predicates the tcgen05 instructions themselves on one elected lane.  Measured on B200 in a
// micro-benchmark: issued from inside a divergent `if (lane == 0)` region, an MMA costs the issuing warp
// enough instruction slots that FMA-bound warps on the same scheduler stretch it from 48 to 122 clocks
// per instruction; issued convergently it stays at the tensor pipe's own 46 clocks.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t el;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(el));
  return el;
}
// A whole K loop in one instruction sequence: NK tensor-core instructions D[tmem] (+)= A_k * B_k, k = 0..NK-1,
// all predicated on `go`, the first one accumulating only if `acc0`.  Operand k is operand 0 moved by a
// compile-time step: for shared-memory operands the low descriptor half advances by step(k) (16-byte units),
// AK / BK select the step pattern (true: K-major tile of two 64-element panels 16 KB apart, 32 bytes per K step
// inside a panel; false: MN-major tile, 2 KB per K step); for a tensor-memory A operand the column advances by
// 16 per K step.  One predicate set-up for the group instead of one per instruction keeps the issuing warp's
// instruction count per MMA at three.
template <bool K_MAJOR>
__host__ __device__ constexpr uint32_t umma_kstep(int k) {
  return K_MAJOR ? (uint32_t)((k >> 2) * 1024 + (k & 3) * 2) : (uint32_t)(k * 128);
}
#define LA_UMMA_SS_STEP(AI, BI)                                  \
  "add.u32 al, %1, " #AI ";\n\tmov.b64 da, {al, %3};\n\t"        \
  "add.u32 bl, %2, " #BI ";\n\tmov.b64 db, {bl, %3};\n\t"        \
  "@g tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, t;\n\t"
template <int NK, bool AK, bool BK>
__device__ __forceinline__ void umma_group_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi,
                                              uint32_t idesc, uint32_t acc0, uint32_t go) {
  static_assert(NK == 4 || NK == 8, "K steps per group");
  if (NK == 8) {
    asm volatile(
        "{\n\t.reg .pred p, g, t;\n\t.reg .b64 da, db;\n\t.reg .b32 al, bl;\n\t"
        "setp.ne.b32 g, %6, 0;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "@g tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t"
        LA_UMMA_SS_STEP(%7, %14) LA_UMMA_SS_STEP(%8, %15) LA_UMMA_SS_STEP(%9, %16) LA_UMMA_SS_STEP(%10, %17)
        LA_UMMA_SS_STEP(%11, %18) LA_UMMA_SS_STEP(%12, %19) LA_UMMA_SS_STEP(%13, %20)
        "}" ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc0), "r"(go),
        "n"(umma_kstep<AK>(1)), "n"(umma_kstep<AK>(2)), "n"(umma_kstep<AK>(3)), "n"(umma_kstep<AK>(4)),
        "n"(umma_kstep<AK>(5)), "n"(umma_kstep<AK>(6)), "n"(umma_kstep<AK>(7)),
        "n"(umma_kstep<BK>(1)), "n"(umma_kstep<BK>(2)), "n"(umma_kstep<BK>(3)), "n"(umma_kstep<BK>(4)),
        "n"(umma_kstep<BK>(5)), "n"(umma_kstep<BK>(6)), "n"(umma_kstep<BK>(7))
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p, g, t;\n\t.reg .b64 da, db;\n\t.reg .b32 al, bl;\n\t"
        "setp.ne.b32 g, %6, 0;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "@g tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t"
        LA_UMMA_SS_STEP(%7, %10) LA_UMMA_SS_STEP(%8, %11) LA_UMMA_SS_STEP(%9, %12)
        "}" ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc0), "r"(go),
        "n"(umma_kstep<AK>(1)), "n"(umma_kstep<AK>(2)), "n"(umma_kstep<AK>(3)),
        "n"(umma_kstep<BK>(1)), "n"(umma_kstep<BK>(2)), "n"(umma_kstep<BK>(3))
        : "memory");
  }
}
#undef LA_UMMA_SS_STEP
// Eight K steps with A in tensor memory (16 columns per step) and an MN-major B tile in shared memory.
#define LA_UMMA_TS_STEP(AI, BI)                                  \
  "add.u32 at, %1, " #AI ";\n\t"                                 \
  "add.u32 bl, %2, " #BI ";\n\tmov.b64 db, {bl, %3};\n\t"        \
  "@g tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, t;\n\t"
__device__ __forceinline__ void umma_group_ts8(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi,
                                               uint32_t idesc, uint32_t acc0, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred p, g, t;\n\t.reg .b64 db;\n\t.reg .b32 at, bl;\n\t"
      "setp.ne.b32 g, %6, 0;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "@g tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t"
      LA_UMMA_TS_STEP(16, 128) LA_UMMA_TS_STEP(32, 256) LA_UMMA_TS_STEP(48, 384) LA_UMMA_TS_STEP(64, 512)
      LA_UMMA_TS_STEP(80, 640) LA_UMMA_TS_STEP(96, 768) LA_UMMA_TS_STEP(112, 896)
      "}" ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc0), "r"(go)
      : "memory");
}
// Eight K steps with a dense A operand in tensor memory (8 columns per step) and a B tile of 128 x 128 in shared
// memory, K-major (BK) or MN-major.
template <bool BK>
__device__ __forceinline__ void umma_group_tsd(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi,
                                               uint32_t idesc, uint32_t acc0, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred p, g, t;\n\t.reg .b64 db;\n\t.reg .b32 at, bl;\n\t"
      "setp.ne.b32 g, %6, 0;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "@g tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t"
      LA_UMMA_TS_STEP(8, %7) LA_UMMA_TS_STEP(16, %8) LA_UMMA_TS_STEP(24, %9) LA_UMMA_TS_STEP(32, %10)
      LA_UMMA_TS_STEP(40, %11) LA_UMMA_TS_STEP(48, %12) LA_UMMA_TS_STEP(56, %13)
      "}" ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc0), "r"(go),
      "n"(umma_kstep<BK>(1)), "n"(umma_kstep<BK>(2)), "n"(umma_kstep<BK>(3)), "n"(umma_kstep<BK>(4)),
      "n"(umma_kstep<BK>(5)), "n"(umma_kstep<BK>(6)), "n"(umma_kstep<BK>(7))
      : "memory");
}
// Four such steps (64 rows of K).
template <bool BK>
__device__ __forceinline__ void umma_group_tsd4(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi,
                                                uint32_t idesc, uint32_t acc0, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred p, g, t;\n\t.reg .b64 db;\n\t.reg .b32 at, bl;\n\t"
      "setp.ne.b32 g, %6, 0;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "mov.b64 db, {%2, %3};\n\t"
      "@g tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t"
      LA_UMMA_TS_STEP(8, %7) LA_UMMA_TS_STEP(16, %8) LA_UMMA_TS_STEP(24, %9)
      "}" ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc0), "r"(go),
      "n"(umma_kstep<BK>(1)), "n"(umma_kstep<BK>(2)), "n"(umma_kstep<BK>(3))
      : "memory");
}
#undef LA_UMMA_TS_STEP
// Four K steps of D[e, i] (+)= A[e, j] B[j, i] where B[j, i] = 0 for i < j (REV: for i > j): step k covers
// j = 16 k .. 16 k + 15 and touches only the columns of D that it can change.  Steps K0, K0 + 1, .. (REV: K0, K0 - 1, ..),
// so that step 0 (REV: 7), which covers every column, comes first.  A is MN-major, B K-major, both in shared memory.
template <int K, bool REV>
struct TriStep {
  static constexpr uint32_t n = REV ? 16 * (K + 1) : 128 - 16 * K;        // columns of D
  static constexpr uint32_t dcol = REV ? 0 : 16 * K;                        // first of them
  static constexpr uint32_t a = K * 128;                                    // 2 KB per 16 tokens
  static constexpr uint32_t b = (K >> 2) * 1024 + (K & 3) * 2 + dcol * 8;  // panel, 32 bytes per step, 128 bytes per row
  static constexpr uint32_t idesc = umma_idesc_bf16(128, n, true, false);
};
#define LA_UMMA_TRI_STEP(DO, AO, BO, ID, PRED)                                              \
  "add.u32 dt, %0, " #DO ";\n\tadd.u32 al, %1, " #AO ";\n\tadd.u32 bl, %2, " #BO ";\n\t"  \
  "mov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\tmov.b32 id, " #ID ";\n\t"           \
  "@g tcgen05.mma.cta_group::1.kind::f16 [dt], da, db, id, " #PRED ";\n\t"
template <int K0, bool REV>
__device__ __forceinline__ void umma_tri4(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t acc0,
                                          uint32_t go) {
  constexpr int S = REV ? -1 : 1;
  using T0 = TriStep<K0, REV>;
  using T1 = TriStep<K0 + S, REV>;
  using T2 = TriStep<K0 + 2 * S, REV>;
  using T3 = TriStep<K0 + 3 * S, REV>;
  asm volatile(
      "{\n\t.reg .pred p, g, t;\n\t.reg .b64 da, db;\n\t.reg .b32 dt, al, bl, id;\n\t"
      "setp.ne.b32 g, %5, 0;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      LA_UMMA_TRI_STEP(%6, %7, %8, %9, p) LA_UMMA_TRI_STEP(%10, %11, %12, %13, t)
      LA_UMMA_TRI_STEP(%14, %15, %16, %17, t) LA_UMMA_TRI_STEP(%18, %19, %20, %21, t)
      "}" ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(acc0), "r"(go),
      "n"(T0::dcol), "n"(T0::a), "n"(T0::b), "n"(T0::idesc), "n"(T1::dcol), "n"(T1::a), "n"(T1::b), "n"(T1::idesc),
      "n"(T2::dcol), "n"(T2::a), "n"(T2::b), "n"(T2::idesc), "n"(T3::dcol), "n"(T3::a), "n"(T3::b), "n"(T3::idesc)
      : "memory");
}
#undef LA_UMMA_TRI_STEP
// Arrives on the mbarrier once all tcgen05.mma issued so far by this thread have completed; takes effect only in lanes with go != 0.
__device__ __forceinline__ void umma_commit_if(uint64_t* bar, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred g;\n\tsetp.ne.b32 g, %1, 0;\n\t"
      "@g tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)),
      "r"(go)
      : "memory");
}

}  // namespace ptx
}  // namespace la
