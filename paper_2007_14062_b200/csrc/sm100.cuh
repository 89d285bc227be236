// Shared pieces of the tensor-core kernels (sm_100a): PTX wrappers for barriers, TMA, tensor memory and tcgen05, bounded
// waits, packed fp32 arithmetic, and the host's tensor maps.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

#include "kernels.h"
#include "../../include/bigbird.h"

namespace bigbird {
namespace {

constexpr int kBlock = 64;                 // tokens per block (b) and head dimension (D)
constexpr int kTileBytes = kBlock * kBlock * 2;      // one 64x64 bf16 tile
constexpr long long kWaitLimitCycles = 4000000000ll;   // about two seconds

// ------------------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Non-blocking test of a phase (for the roles that poll several barriers).
__device__ __forceinline__ bool mbar_test(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// One thread of a converged warp.  (An MMA issued behind "lane == 0" instead costs more to issue: the gradients of the base workload
// took 857 us so and 557 us from an elected thread.)
__device__ __forceinline__ bool elect_one() {
    unsigned e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}

// Bounded wait, small enough to sit inline at every site (the kernel's hot code has to fit the SM's instruction
// cache, measured at between 32 and 48 KB: a loop with a clock read and its own give-up code per site did not).  A
// failing try keeps the thread suspended for about 1.4 us on this part (measured); after kWaitTries of them, about
// two seconds, the wait is abandoned.  Returns false then, or as soon as another
// thread of the CTA has given up; the caller leaves its loop and calls give_up with the code of the wait.
constexpr unsigned kWaitTries = 1500000;
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, int* abort_flag) {
    // a phase that is already complete is seen by the plain test in a dozen cycles; try_wait, which may put the
    // thread to sleep, takes a few hundred even then (measured on the MMA thread's time line)
    if (mbar_test(bar, parity)) return true;
#pragma unroll 1
    for (unsigned it = 0; it < kWaitTries; ++it) {
        if (mbar_try(bar, parity)) return true;
        if (*(volatile int*)abort_flag) break;
    }
    return false;
}
// Records BIGBIRD_ETIMEOUT and the code of the abandoned wait (the first one wins) and tells the rest of the CTA.
__device__ __forceinline__ void give_up(int* abort_flag, int* status, int code) {
    if (*(volatile int*)abort_flag == 0) {
        if (atomicCAS(status, 0, BIGBIRD_ETIMEOUT) == 0) status[1] = code;
        *(volatile int*)abort_flag = 1;
    }
}
// Checked build (-DBB_DEBUG): indices that come out of the schedule are tested against their ranges before they are
// used as addresses; a failing check records BIGBIRD_EINTERNAL with its code, tells the CTA to stop, and the access
// is skipped.  Nothing traps.  (The memory checker is not available where this library is developed; small cases
// against the oracle and this build stand in for it.)
#ifdef BB_DEBUG
__device__ __forceinline__ bool debug_check(bool good, int* abort_flag, int* status, int code) {
    if (!good && *(volatile int*)abort_flag == 0) {
        if (atomicCAS(status, 0, BIGBIRD_EINTERNAL) == 0) status[1] = code;
        *(volatile int*)abort_flag = 1;
    }
    return good;
}
#define BB_CHECK(cond, code) debug_check((cond), &ctl->abort_flag, p.status, (code))
#else
#define BB_CHECK(cond, code) true
#endif

// The same bound for a role that polls: tick() is called whenever a round over the role's barriers found nothing
// to do; it backs off (a polling warp that spins takes issue slots from the softmax warps of its sub-partition)
// and returns false once the CTA has given up or the idle time exceeds the limit.
struct IdleClock {
    unsigned n = 0;
    long long t0 = 0;
    __device__ __forceinline__ void reset() { n = 0; }
    __device__ __forceinline__ bool tick(int* abort_flag, int* status, int code, unsigned sleep_ns) {
        ++n;
        if ((n & 15u) == 0u) {
            if (*(volatile int*)abort_flag) return false;
            const long long now = clock64();
            if (n == 16u) t0 = now;
            else if (now - t0 > kWaitLimitCycles) {
                give_up(abort_flag, status, code);
                return false;
            }
        }
        if (sleep_ns) __nanosleep(sleep_ns);
        return true;
    }
};

__device__ __forceinline__ void tma_load_tile(void* dst, const CUtensorMap* tm, int row, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"((unsigned long long)tm), "r"(0), "r"(row), "r"(smem_u32(bar)) : "memory");
}
// Writes a 64 x 64 tile from shared memory (128-byte swizzle) to the rows of a tensor map's tensor.
__device__ __forceinline__ void tma_store_tile(const CUtensorMap* tm, int row, const void* src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"((unsigned long long)tm), "r"(0), "r"(row), "r"(smem_u32(src)) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// Read where the program says so: behind the barrier tests that come before it.
__device__ __forceinline__ unsigned ld_shared(const unsigned* p) {
    unsigned v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_shared16(unsigned addr, unsigned a, unsigned b, unsigned c, unsigned d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Untiled copy: both addresses and the size are multiples of 16 bytes.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"((unsigned long long)__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(unsigned d_tmem, unsigned long long a_desc, unsigned long long b_desc, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(unsigned d_tmem, unsigned a_tmem, unsigned long long b_desc, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

// The same, issued only if enable != 0 (a predicated instruction instead of a branch around it: a lone thread pays
// for every branch it executes with a stall until the target is known).
__device__ __forceinline__ void mma_ts_if(unsigned d_tmem, unsigned a_tmem, unsigned long long b_desc, unsigned idesc, unsigned accumulate, unsigned enable) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(enable) : "memory");
}
__device__ __forceinline__ void tc_commit_if(unsigned long long* bar, unsigned enable) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(smem_u32(bar)), "r"(enable) : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle, 8-row groups 1024 bytes apart (a dense 64-wide bf16 tile).
__device__ __forceinline__ unsigned long long smem_desc_sw128(unsigned addr) {
    return (unsigned long long)((addr & 0x3FFFFu) >> 4)
         | (1ull << 16)                       // leading byte offset (unused for a single 128-byte atom)
         | ((unsigned long long)(1024 >> 4) << 32)   // stride byte offset: next group of 8 rows
         | (1ull << 46)                       // descriptor version of sm_100
         | (2ull << 61);                      // SWIZZLE_128B
}
// The same by its low word (the high word is the same for every such tile).
constexpr unsigned kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ unsigned smem_desc_lo(unsigned addr) { return ((addr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ void mma_ss_lo(unsigned d_tmem, unsigned a_lo, unsigned b_lo, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi) : "memory");
}
__device__ __forceinline__ void mma_ts_lo(unsigned d_tmem, unsigned a_tmem, unsigned b_lo, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\tmov.b64 b, {%2, %5};\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi) : "memory");
}
// The same, leaving lanes 0..63 or 64..127 of D as they are: skip_upper and skip_lower are all ones or zero.
__device__ __forceinline__ void mma_ss_half(unsigned d_tmem, unsigned a_lo, unsigned b_lo, unsigned idesc, unsigned accumulate,
                                            unsigned skip_upper, unsigned skip_lower) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, {%6, %6, %7, %7}, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi), "r"(skip_upper), "r"(skip_lower) : "memory");
}
__device__ __forceinline__ void mma_ts_half(unsigned d_tmem, unsigned a_tmem, unsigned b_lo, unsigned idesc, unsigned accumulate,
                                            unsigned skip_upper, unsigned skip_lower) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\tmov.b64 b, {%2, %5};\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %3, {%6, %6, %7, %7}, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi), "r"(skip_upper), "r"(skip_lower) : "memory");
}
// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = 64 (Q K^T adds 64 per further key block); B is K-major (K^T) or MN-major (V).
constexpr unsigned kIdescQK64 = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);   // N field (bits 17..22) = N / 8
constexpr unsigned kIdescPV = kIdescQK64 | (1u << 16);

#define BB_REP32(F, o) F(o+0), F(o+1), F(o+2), F(o+3), F(o+4), F(o+5), F(o+6), F(o+7), F(o+8), F(o+9), F(o+10), F(o+11), \
    F(o+12), F(o+13), F(o+14), F(o+15), F(o+16), F(o+17), F(o+18), F(o+19), F(o+20), F(o+21), F(o+22), F(o+23), \
    F(o+24), F(o+25), F(o+26), F(o+27), F(o+28), F(o+29), F(o+30), F(o+31)
#define BB_OUT(i) "=r"(u[i])
#define BB_IN(i) "r"(u[i])
__device__ __forceinline__ void tmem_ld64(unsigned taddr, float* r) {
    unsigned* u = reinterpret_cast<unsigned*>(r);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
        "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
        "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];"
        : BB_REP32(BB_OUT, 0), BB_REP32(BB_OUT, 32) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld32(unsigned taddr, float* r) {
    unsigned* u = reinterpret_cast<unsigned*>(r);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : BB_REP32(BB_OUT, 0) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(unsigned taddr, const unsigned* u) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
        ::BB_REP32(BB_IN, 0), "r"(taddr) : "memory");
}
#define BB_REP16(F, o) F(o+0), F(o+1), F(o+2), F(o+3), F(o+4), F(o+5), F(o+6), F(o+7), F(o+8), F(o+9), F(o+10), F(o+11), \
    F(o+12), F(o+13), F(o+14), F(o+15)
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float* r) {
    unsigned* u = reinterpret_cast<unsigned*>(r);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : BB_REP16(BB_OUT, 0) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(unsigned taddr, const unsigned* u) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
        ::BB_REP16(BB_IN, 0), "r"(taddr) : "memory");
}
#undef BB_OUT
#undef BB_IN
__device__ __forceinline__ void tmem_st32_zero(unsigned taddr) {
    const unsigned z = 0;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%1], "
        "{%0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, "
        "%0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0, %0};"
        ::"r"(z), "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
    unsigned d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// (x0, x1) * a + b on the packed fp32 pipe
__device__ __forceinline__ void ffma2(float& r0, float& r1, float x0, float x1, float a, float b) {
    asm("{ .reg .b64 ra, rb, rc, rd; mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %4}; mov.b64 rc, {%5, %5}; "
        "fma.rn.f32x2 rd, ra, rb, rc; mov.b64 {%0, %1}, rd; }"
        : "=f"(r0), "=f"(r1) : "f"(x0), "f"(x1), "f"(a), "f"(b));
}
__device__ __forceinline__ void fadd2(float& r0, float& r1, float x0, float x1) {
    asm("{ .reg .b64 ra, rb, rd; mov.b64 ra, {%0, %1}; mov.b64 rb, {%2, %3}; add.f32x2 rd, ra, rb; mov.b64 {%0, %1}, rd; }"
        : "+f"(r0), "+f"(r1) : "f"(x0), "f"(x1));
}
__device__ __forceinline__ void fmul2(float& r0, float& r1, float a) {
    asm("{ .reg .b64 ra, rb, rd; mov.b64 ra, {%0, %1}; mov.b64 rb, {%2, %2}; mul.f32x2 rd, ra, rb; mov.b64 {%0, %1}, rd; }"
        : "+f"(r0), "+f"(r1) : "f"(a));
}
// (x0, x1) * a + (b0, b1)
__device__ __forceinline__ void ffma2v(float& r0, float& r1, float x0, float x1, float a, float b0, float b1) {
    asm("{ .reg .b64 ra, rb, rc, rd; mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %4}; mov.b64 rc, {%5, %6}; "
        "fma.rn.f32x2 rd, ra, rb, rc; mov.b64 {%0, %1}, rd; }"
        : "=f"(r0), "=f"(r1) : "f"(x0), "f"(x1), "f"(a), "f"(b0), "f"(b1));
}
// ((x0, x1) + (b0, b1)) * (p0, p1)
__device__ __forceinline__ void add_mul2(float& r0, float& r1, float x0, float x1, float b0, float b1, float p0, float p1) {
    asm("{ .reg .b64 ra, rb, rc, rd; mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %5}; mov.b64 rc, {%6, %7}; "
        "add.rn.f32x2 rd, ra, rb; mul.rn.f32x2 rd, rd, rc; mov.b64 {%0, %1}, rd; }"
        : "=f"(r0), "=f"(r1) : "f"(x0), "f"(x1), "f"(b0), "f"(b1), "f"(p0), "f"(p1));
}
// (x0, x1) as a sum of two pairs of bf16: hi the values rounded to bf16, lo what that leaves, rounded in turn (16
// significant bits together)
__device__ __forceinline__ void split_bf16(float x0, float x1, unsigned& hi, unsigned& lo) {
    hi = pack_bf16(x0, x1);
    const float h0 = __uint_as_float(hi << 16), h1 = __uint_as_float(hi & 0xffff0000u);
    lo = pack_bf16(x0 - h0, x1 - h1);
}

// ------------------------------------------------------------------------------------------------ host side
// A launch that may begin before the kernel in front of it in the stream has drained; the kernel waits for it itself.
template <typename... Ps, typename... As>
cudaError_t launch_chained(void (*kernel)(Ps...), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream, const As&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, Ps(args)...);
}
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)sym;
    });
    return fn;
}

// [rows, 64] bf16 row-major tensor read (or written) in boxes of 64 rows with the 128-byte swizzle.
inline bool make_map(CUtensorMap* tm, const void* base, uint64_t rows) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)kBlock, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(kBlock * 2)};
    cuuint32_t box[2] = {(cuuint32_t)kBlock, (cuuint32_t)kBlock};
    cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace
}  // namespace bigbird
