// Device primitives shared by the de-dispersion kernels: mbarriers with
// bounded waits, TMA bulk copies, byte permutes and adds, tensor-memory
// accesses.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "dd_internal.h"

namespace dd {
namespace {

constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t mb, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx_arrive(uint32_t mb, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mb, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.shared::cta.b64 [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mb) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t mb, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; "
        "selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(mb), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the completion of the phase with the given parity.  The
// waiting warp backs off with __nanosleep (64 ns doubling to 1 us) so it does
// not take issue slots from the warps that share its scheduler; the global
// timer is read every 16 tries.
__device__ __noinline__ bool mbar_wait_slow(uint32_t mb, uint32_t parity, uint64_t limit_ns) {
    const uint64_t t0 = global_ns();
    uint32_t ns = 64;
    for (uint32_t i = 1;; ++i) {
        if (mbar_try(mb, parity))
            return true;
        __nanosleep(ns);
        ns = ns < 1024u ? 2u * ns : 1024u;
        if ((i & 15u) == 0 && global_ns() - t0 > limit_ns)
            return false;
    }
}

__device__ __forceinline__ bool mbar_wait(uint32_t mb, uint32_t parity,
                                          uint64_t limit_ns = kWaitLimitNs) {
    return mbar_try(mb, parity) || mbar_wait_slow(mb, parity, limit_ns);
}

// The same in line and without the back-off, for kernels that wait in the
// steady state and split their registers between warps (ptxas does not allow
// a call there).
__device__ __forceinline__ bool mbar_spin(uint32_t mb, uint32_t parity) {
    if (mbar_try(mb, parity))
        return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try(mb, parity))
        if (global_ns() - t0 > kWaitLimitNs)
            return false;
    return true;
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes,
                                         uint32_t mb) {
    asm volatile(
        "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            dst),
        "l"(src), "r"(bytes), "r"(mb)
        : "memory");
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// acc + p on the FMA pipe (p * one + acc with one == 1 at run time).
__device__ __forceinline__ uint32_t imad_acc(uint32_t p, uint32_t one, uint32_t acc) {
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(p), "r"(one), "r"(acc));
    return r;
}

__device__ __forceinline__ int shift_of(float dm, float ds) {
    return __float2int_rz(__fmul_rn(dm, ds));
}

__device__ __forceinline__ float add_f16_lo(uint32_t x, float acc) {
    float r;
    asm("{ .reg .b16 lo, hi; mov.b32 {lo, hi}, %1; add.rn.f32.f16 %0, lo, %2; }"
        : "=f"(r)
        : "r"(x), "f"(acc));
    return r;
}

__device__ __forceinline__ float add_f16_hi(uint32_t x, float acc) {
    float r;
    asm("{ .reg .b16 lo, hi; mov.b32 {lo, hi}, %1; add.rn.f32.f16 %0, hi, %2; }"
        : "=f"(r)
        : "r"(x), "f"(acc));
    return r;
}

__device__ __forceinline__ void record(int *status, int code) {
    atomicCAS(status, kDevOk, code);
}

// Tensor-memory (TMEM) access of one warp: N consecutive 32-bit columns of
// its 32 lanes (thread i: lane i).  The FP16/FP32 consumers keep their
// running sums and compensations there (written and read once per block of
// channels).
template <int N>
__device__ __forceinline__ void tm_ld(uint32_t taddr, uint32_t (&v)[N]) {
    static_assert(N == 4 || N == 8 || N == 16, "TMEM load width");
    if constexpr (N == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                     : "r"(taddr)
                     : "memory");
    else if constexpr (N == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, "
                     "[%8];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                       "=r"(v[6]), "=r"(v[7])
                     : "r"(taddr)
                     : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, "
                     "%8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                       "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
                       "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                     : "r"(taddr)
                     : "memory");
}

template <int N>
__device__ __forceinline__ void tm_st(uint32_t taddr, const uint32_t (&v)[N]) {
    static_assert(N == 4 || N == 8 || N == 16, "TMEM store width");
    if constexpr (N == 4)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr),
                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
                     : "memory");
    else if constexpr (N == 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, "
                     "%8};" ::"r"(taddr),
                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]),
                     "r"(v[7])
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, "
                     "%8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]),
                     "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]),
                     "r"(v[13]), "r"(v[14]), "r"(v[15])
                     : "memory");
}

__device__ __forceinline__ void tm_wait_ld() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tm_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Registers written by tcgen05.ld hold their values only after
// tcgen05.wait::ld, which the compiler does not know: after each wait the
// loaded registers pass through an empty volatile asm that redefines them, so
// no use of them can be scheduled above the wait.
template <int N>
__device__ __forceinline__ void reg_fence(uint32_t (&v)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i)
        asm volatile("" : "+r"(v[i]));
}

}  // namespace
}  // namespace dd
