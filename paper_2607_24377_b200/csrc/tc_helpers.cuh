// tcgen05 / mbarrier / bulk-copy helpers shared by the attention kernels (sm_100a, inline PTX).
#pragma once
#include <type_traits>

#include "common.cuh"

namespace mxattn {
namespace fwd {

// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Explicit shared-space accesses with 32-bit addresses (no generic-pointer arithmetic).
__device__ __forceinline__ void sts128(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ void sts32f(uint32_t addr, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ float lds32f(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// Two fused multiply-adds in one instruction (packed fp32x2): (a0, a1) * cc + dd with cc = (c, c), dd = (d, d);
// each half is an IEEE fp32 fma, bit-identical to fmaf.
__device__ __forceinline__ uint64_t dup2(float v) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ void fma2(uint32_t a0_bits, uint32_t a1_bits, uint64_t cc, uint64_t dd, float& r0, float& r1) {
  uint64_t ab, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ab) : "r"(a0_bits), "r"(a1_bits));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(ab), "l"(cc), "l"(dd));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r0), "=f"(r1) : "l"(r));
}
// (a0 + a2) + (a4 + a6) and (a1 + a3) + (a5 + a7) with three packed fp32x2 additions (each half an IEEE fp32 add)
__device__ __forceinline__ void add2x2(float a0, float a1, float a2, float a3, float a4, float a5, float a6, float a7,
                                       float& r0, float& r1) {
  uint64_t p0, p1, p2, p3, q0, q1, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p0) : "f"(a0), "f"(a1));
  asm("mov.b64 %0, {%1, %2};" : "=l"(p1) : "f"(a2), "f"(a3));
  asm("mov.b64 %0, {%1, %2};" : "=l"(p2) : "f"(a4), "f"(a5));
  asm("mov.b64 %0, {%1, %2};" : "=l"(p3) : "f"(a6), "f"(a7));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(q0) : "l"(p0), "l"(p1));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(q1) : "l"(p2), "l"(p3));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(q0), "l"(q1));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r0), "=f"(r1) : "l"(r));
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  // the third operand is a suspend-time hint (ns): the thread sleeps in hardware instead of spinning
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {     // non-blocking
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}

// Bounded wait.  Returns false if the wait was abandoned (own limit reached, or another thread of
// the CTA already gave up); the caller then skips to the teardown.
constexpr long long kWaitLimitCycles = 4000000000LL;   // ~2 s at full clock
// `abort_flag` is the flag the wait watches; `raise_flag`, if given, is the one it sets on expiry instead.
__device__ __forceinline__ bool mbar_wait_loop(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int* status, int code, long long limit, volatile int* raise_flag) {
  const long long t0 = clock64();
  for (int it = 1;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 15) == 0) {
      if (*abort_flag) return false;
      if (clock64() - t0 > limit) {
        *(raise_flag ? raise_flag : abort_flag) = 1;
        atomicCAS(status, 0, code);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, int code, long long limit = kWaitLimitCycles,
                                          volatile int* raise_flag = nullptr) {
  if (mbar_try(bar, parity)) return true;
  return mbar_wait_loop(bar, parity, abort_flag, status, code, limit, raise_flag);
}
// The same wait with its loop out of line, for the single-thread roles (copy producer, MMA issuer): their time per
// tile grows with the amount of code they walk through, not only with the instructions they execute, and this keeps
// one try_wait and a branch per wait in their loops.  (In the softmax warps, which run at the register limit, the
// call's register conventions cost more than the compact code gains.)
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                   int* status, int code) {
  return mbar_wait_loop(bar, parity, abort_flag, status, code, kWaitLimitCycles, nullptr);
}
__device__ __forceinline__ bool mbar_wait1(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code) {
  if (mbar_try(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, abort_flag, status, code);
}

// Two warps that share query rows (each holds half of the key columns) meet at a 64-thread named barrier to exchange
// a value per row.  A warp that has given up on its own work (a bounded wait ran out) must not simply leave, because
// its partner may already be on its way to the next meeting; it keeps the remaining `n` appointments and does nothing
// else.  Kept out of line: it is never executed in a healthy run.
static __device__ __noinline__ void pair_keep_company(int pair_bar, int n) {
  for (int i = 0; i < n; ++i) asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// ---------------------------------------------------------------------------------------------
// An MMA issuer that runs as a converged warp: all its lanes walk the loop, so that loop counters, addresses and descriptors
// live in uniform registers, and one elected lane issues each tcgen05 instruction under a predicate.  In code that only
// one lane executes, every descriptor word is moved from a vector to a uniform register in front of each instruction
// (about 100 cycles per tcgen05 instruction).
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0); }   // uniform for the compiler too
// The thread index read afresh: what an epilogue derives from it does not occupy registers during the loop before.
__device__ __forceinline__ uint32_t fresh_tid() { uint32_t v; asm volatile("mov.u32 %0, %%tid.x;" : "=r"(v)); return v; }
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r;
}
static __device__ __noinline__ bool mbar_wait_warp_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code) {
  return __all_sync(0xFFFFFFFFu, mbar_wait_loop(bar, parity, abort_flag, status, code, kWaitLimitCycles, nullptr));
}
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code) {
  if (__all_sync(0xFFFFFFFFu, mbar_try(bar, parity))) return true;
  return mbar_wait_warp_slow(bar, parity, abort_flag, status, code);
}
__device__ __forceinline__ void tc_cp_sf_if(uint32_t leader, uint32_t taddr, uint32_t saddr) {
  const uint64_t d = ((uint64_t)((128u >> 4) | (1u << 14)) << 32) | (saddr >> 4);
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t"
               "@p tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;\n\t}" ::"r"(taddr), "l"(d), "r"(leader) : "memory");
}
__device__ __forceinline__ void tc_commit_if(uint32_t leader, uint32_t bar) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\t"
               "@p tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(leader) : "memory");
}
__device__ __forceinline__ void tc_mma_if(uint32_t leader, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
               "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb), "r"(leader) : "memory");
}

__device__ __forceinline__ void tc_cp_sf(uint32_t taddr, uint32_t saddr) {   // 512-byte scale atom -> 4 columns
  const uint64_t d = ((uint64_t)((128u >> 4) | (1u << 14)) << 32) | (saddr >> 4);   // no swizzle, 8-row groups 128 B apart
  asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(d) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// ---------------------------------------------------------------------------------------------
// instruction descriptor of kind::mxf4.block_scale: A, B = E2M1 (K-major), scales UE8M0, M = 128
__device__ __forceinline__ constexpr uint32_t make_idesc(int n, int ks) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((128u >> 4) << 24) |
         ((uint32_t)(ks * 2) << 29) | ((uint32_t)(ks * 2) << 4);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
               ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The attention kernels allocate all 512 columns, so that their tensor memory starts at column 0, and address it from there.
// Were it ever elsewhere, this code in the status word says that the output is void.  Where a CTA's abort flag reaches the
// status word at its end, the flag takes it at the start (2 x 1024: no time; at the end it took 0.1 of 10.6 us); elsewhere the
// warp that allocated checks at the end (in front of the loops it costs registers: NVFP4 direct, 40 x 16384, 3860 -> 4070 us).
constexpr int kCodeTmemBase = 41;
__device__ __forceinline__ void check_tmem_base(uint32_t base, int lane, int* status) {
  if (base != 0u && lane == 0) atomicCAS(status, 0, kCodeTmemBase);
}

#define TMEM_LD32(taddr, r)                                                                                   \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "                                                      \
               "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,"  \
               "%25,%26,%27,%28,%29,%30,%31}, [%32];"                                                         \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),          \
                 "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),      \
                 "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),   \
                 "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),   \
                 "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])                                           \
               : "r"(taddr) : "memory")

#define TMEM_LD64(taddr, r)  \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];" \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]) \
               : "r"(taddr) : "memory")

#define TMEM_ST32(taddr, r)                                                                                   \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "                                               \
               "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,"  \
               "%25,%26,%27,%28,%29,%30,%31};"                                                                \
               ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),      \
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),\
                 "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]),          \
                 "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),          \
                 "r"(r[30]), "r"(r[31]), "r"(taddr) : "memory")

#define TMEM_LD16(taddr, r)                                                                                   \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];" \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), \
                 "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr) : "memory")
#define TMEM_ST16(taddr, r)                                                                                   \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" \
               ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), \
                 "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr) : "memory")
#define TMEM_LD8(taddr, r)                                                                            \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"              \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) \
               : "r"(taddr) : "memory")
#define TMEM_ST8(taddr, r)                                                                            \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"              \
               ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr) : "memory")

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// tcgen05.wait::ld that names registers of the loads it waits for, so that no use of them can move ahead of it
#define TMEM_LD_WAIT32(r)                                                                                              \
  asm volatile("tcgen05.wait::ld.sync.aligned;"                                                                        \
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),       \
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), \
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]),            \
                 "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),            \
                 "+r"(r[30]), "+r"(r[31])::"memory")
#define TMEM_LD_WAIT16(r)                                                                                              \
  asm volatile("tcgen05.wait::ld.sync.aligned;"                                                                        \
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),       \
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory")
// Keys beyond the sequence do not exist: the scores of columns `valid` to `cols` - 1 (of this warp's 32 rows, at `taddr`) become
// -inf in tensor memory, before the warp loads its scores.  Replacing them in the registers behind the load costs every tile,
// not only the last: the values of both paths have to meet in one set of registers, which the load's own consecutive ones are
// not, and the compiler copies all of them: 1548 -> 1411 cycles per tile in an early build of walk.cuh (one team, no rescaling), of
// which every instruction of a tile is seen.  (The kernel of forward.cu gets slower, 61.6 -> 64.1 ms at 40 x 75600, so the others mask their registers.)
__device__ __forceinline__ void mask_scores(uint32_t taddr, int valid, int cols) {
  int i = valid < 0 ? 0 : valid;
#pragma unroll 1
  for (; i < cols && (i & 7) != 0; ++i)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr + i), "r"(0xFF800000u) : "memory");
#pragma unroll 1
  for (; i < cols; i += 8)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr + i), "r"(0xFF800000u) : "memory");
  tmem_st_wait();
}
__device__ __forceinline__ int lds_volatile(uint32_t addr) {
  int v;
  asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
// A wait after which the caller goes on in any case: it gives up on its own limit (about two seconds; the code then goes
// into the CTA's abort flag, from where it reaches `status` at the end) or when the abort flag is up; every later wait of the
// CTA then returns when its try_wait does, after 4 us.  For warps that meet at named barriers: none of them leaves its loop
// without keeping what meetings are left, so none can be stranded there.  (The flag read in front of the try_wait costs every
// wait that is not satisfied yet, 2 x 1024: 10.6 -> 10.9 us; a shorter time limit for the try_wait is not heeded.)
// kTest: a test_wait in front (a wait that is already satisfied takes 38 cycles as that, 78 as a try_wait).  kOff: of the
// barrier from `bar`.
#define MBAR_SOFT_WAIT(first)                                                        \
  asm volatile("{\n\t.reg .pred p;\n\t.reg .u64 t0, t1;\n\t.reg .u32 a;\n\t" first     \
               "mbarrier.try_wait.parity.shared::cta.b64 p, [%0+%4], %1, 20000;\n\t" \
               "vote.sync.all.pred p, p, 0xffffffff;\n\t"                            \
               "@p bra.uni DONE;\n\t"                                                \
               "mov.u64 t0, %%clock64;\n"                                            \
               "AGAIN:\n\t"                                                          \
               "ld.volatile.shared.u32 a, [%2];\n\t"                                 \
               "setp.ne.u32 p, a, 0;\n\t"                                            \
               "vote.sync.any.pred p, p, 0xffffffff;\n\t"                            \
               "@p bra.uni DONE;\n\t"                                                \
               "mbarrier.try_wait.parity.shared::cta.b64 p, [%0+%4], %1, 20000;\n\t" \
               "vote.sync.all.pred p, p, 0xffffffff;\n\t"                            \
               "@p bra.uni DONE;\n\t"                                                \
               "mov.u64 t1, %%clock64;\n\t"                                          \
               "sub.u64 t1, t1, t0;\n\t"                                             \
               "setp.lt.u64 p, t1, %5;\n\t"                                          \
               "vote.sync.any.pred p, p, 0xffffffff;\n\t"                            \
               "@p bra.uni AGAIN;\n\t"                                               \
               "st.volatile.shared.u32 [%2], %3;\n"                                  \
               "DONE:\n\t}"                                                          \
               ::"r"(bar), "r"(parity), "r"(abort_addr), "n"(kCode), "n"(kOff), "n"(kLimit) : "memory")
template <int kCode, int kOff = 0, bool kTest = false, long long kLimit = kWaitLimitCycles>
__device__ __forceinline__ void mbar_wait_soft(uint32_t bar, uint32_t parity, uint32_t abort_addr) {
  // one block of assembly, so that the usual case is a probe, a vote and a branch, and the rest costs no registers
  if constexpr (kTest)
    MBAR_SOFT_WAIT("mbarrier.test_wait.parity.shared::cta.b64 p, [%0+%4], %1;\n\tvote.sync.all.pred p, p, 0xffffffff;\n\t@p bra.uni DONE;\n\t");
  else
    MBAR_SOFT_WAIT("");
}
#undef MBAR_SOFT_WAIT
// Two teams of softmax warps take the tiles 0 .. F - 1 of a CTA in turn (team t: t, t + 2, ...).  The four warps of a row quarter
// meet once per tile at a named barrier of the team whose tile it is (its two warps wait, the other team's two only arrive,
// behind their own tile's).  Every 64 tiles a warp looks whether the CTA has given up, and then keeps the meetings only: with
// the waits of all tiles that are left, 4 us each, a call would take several times its own time to end.
__device__ __forceinline__ void team_meetings(int f, int F, int own_bar, int other_bar) {
#pragma unroll 1
  for (; f < F; f += 2) {
    asm volatile("bar.sync %0, 128;" ::"r"(own_bar) : "memory");
    asm volatile("bar.arrive %0, 128;" ::"r"(other_bar) : "memory");
  }
}
template <typename Tile, typename Leave>
__device__ __forceinline__ void team_tiles(int t, int F, uint32_t abort_addr, int own_bar, int other_bar, Tile&& tile, Leave&& leave) {
  int f = t;
  for (; f < F; f += 4) {
    if ((f & 60) == 0 && lds_volatile(abort_addr) != 0) {
      leave(f);
      break;
    }
    tile(std::integral_constant<int, 0>{});
    if (f + 2 >= F) return;
    tile(std::integral_constant<int, 1>{});
  }
  team_meetings(f, F, own_bar, other_bar);
}

// 2^x for values that are only rounded to E2M1 (row sum from the quantized probabilities).  The rounding changes at seven values,
// 1/4, 3/4, 5/4, 7/4, 5/2, 7/2 and 5; the polynomial goes through 2^x there and at x = -4, and stays on the same side in between: its
// error, up to 0.0065 between -4 and -2 and below 3e-4 from there to the last change, changes no code.  Below -4 it is less than 2^x and in the end negative (odd degree), which the conversion takes to
// code 0, above the last point more than 5 (codes end at 6).  The coefficients' last places are chosen so that the codes are those
// of ex2.approx for every one of the 2^32 arguments (mxattn_selftest_exp2_codes compares them; in the rounding that the interpolation gives they differ at five).
__device__ __forceinline__ void exp2_poly(float& a, float& b) {
  constexpr float kExp2Poly[8] = {1.00000691f, 0.693127513f, 0.240191191f, 0.0556160808f,
                                  0.00956740882f, 0.00130120874f, 0.000174282599f, 1.70464209e-05f};
  uint64_t x, y;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a), "f"(b));
  y = dup2(kExp2Poly[7]);
#pragma unroll
  for (int i = 6; i >= 0; --i) asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(y) : "l"(y), "l"(x), "l"(dup2(kExp2Poly[i])));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(y));
}
__device__ __forceinline__ uint32_t pack_e2m1x8_relu(float x0, float x1, float x2, float x3, float x4, float x5, float x6, float x7) {
  uint32_t out;
  asm("{\n\t"
      ".reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};\n\t"
      "}"
      : "=r"(out)
      : "f"(x0), "f"(x1), "f"(x2), "f"(x3), "f"(x4), "f"(x5), "f"(x6), "f"(x7));
  return out;
}
__device__ __forceinline__ void sts8(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// (a0, a1) * ss, two IEEE fp32 multiplications in one instruction
__device__ __forceinline__ void mul2(uint32_t& a0, uint32_t& a1, uint64_t ss) {
  uint64_t ab, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ab) : "r"(a0), "r"(a1));
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(ab), "l"(ss));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a0), "=r"(a1) : "l"(r));
}

// Epilogue of a softmax warp: 32 rows x 64 columns of the accumulator at `taddr` times inv_l, to shared memory and from there
// to global memory as tensor copies (boxes of 32 rows x 128 bytes: 64 bf16 columns or 32 fp32 ones, so that fp32 takes two
// turns with the box; rows at or beyond Nq are clipped by the copy).  Written from registers, a warp's 16-byte stores land 256
// or 512 bytes apart (one partly filled sector per lane and instruction), and any store instruction of these warps queues in
// front of the next tile's shared-memory traffic.  The box uses the 128-byte swizzle (16-byte chunk c of row r sits at chunk
// c ^ (r & 7)), which also spreads a quarter warp's stores over all banks.  In the MXFP4 kernel fp32 takes 834 us for 40 x
// 75600 x 512 (1208 from registers), 64.5 for 40 x 4096 x 512 (86), 20.6 for 14 x 1300 x 777 (23.4).
// `box` is 1024-byte aligned; `inside`: whether the first row exists.  The caller waits (cp.async.bulk.wait_group.read in lane
// 0) before the box is used again or the CTA ends.
constexpr int kOutBoxBytes = 32 * 128;
template <bool kOutF32>
__device__ __forceinline__ void store_half_rows(uint32_t taddr, uint32_t box, int lane, float inv_l, const CUtensorMap* map, int col, int row0, int bh, bool inside) {
  const uint32_t aRow = box + lane * 128;
#pragma unroll 1
  for (int c0 = 0; c0 < 64; c0 += 32) {
    uint32_t r32[32];
    TMEM_LD32(taddr + c0, r32);
    if (kOutF32 && c0 > 0) {                         // the first half has left the box
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
    }
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < (kOutF32 ? 8 : 4); ++i) {
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (kOutF32) {
          w[k] = __float_as_uint(__uint_as_float(r32[4 * i + k]) * inv_l);
        } else {
          const float a = __uint_as_float(r32[(8 * i + 2 * k) & 31]) * inv_l, b = __uint_as_float(r32[(8 * i + 2 * k + 1) & 31]) * inv_l;
          asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(b), "f"(a));
        }
      }
      sts128(aRow + ((((kOutF32 ? 0 : c0 >> 3) + i) ^ (lane & 7)) << 4), make_uint4(w[0], w[1], w[2], w[3]));
    }
    if (kOutF32 || c0 > 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0 && inside) {
        asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                     ::"l"(map), "r"(col + (kOutF32 ? c0 : 0)), "r"(row0), "r"(bh), "r"(box) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
    }
  }
}

}  // namespace fwd
}  // namespace mxattn
