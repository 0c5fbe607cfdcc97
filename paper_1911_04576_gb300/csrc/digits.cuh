// Exact integer digits on the tensor cores: what their kernels share.
//
// A number is cut into 7 balanced base-256 digits of a 55-bit integer below one
// power of two per matrix row and per vector; digits are exact in FP16, sums of
// their products exact in FP32 below 2^24 (slices.cu: products of the lattice
// operator, slab_lu.cu: elimination of the macromodels' interior unknowns).
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace emsurf {
namespace {

constexpr int kSl = 7;                       // digits
constexpr int kSlWait = 1 << 16;             // tries of a bounded wait (1.3 s)
// |I_a I_b| <= 2^108 = 2^52 units of level 5, so re +- im sums of up to kSlExact
// sources stay inside int64; beyond, the integers lose a bit per factor of 4
constexpr int kSlExact = 990, kSlMaxN = 7000;   // the latter: two vectors in shared memory

__device__ __forceinline__ uint32_t sl_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void sl_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sl_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void sl_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sl_addr(bar)) : "memory");
}
__device__ __forceinline__ void sl_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sl_addr(bar)), "r"(bytes) : "memory");
}
// one try of a wait; suspends the thread for up to 20 us (re-polling warps slow
// every barrier of the block down)
__device__ __forceinline__ uint32_t sl_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(sl_addr(bar)), "r"(parity), "r"(20000u)
        : "memory");
    return ok;
}
// bounded wait of a single thread
__device__ __forceinline__ bool sl_wait(uint64_t* bar, uint32_t parity, int tries) {
    for (int it = 0; it < tries; ++it)
        if (sl_try(bar, parity)) return true;
    return false;
}
// Bounded wait of a whole warp: every try is voted on, so that the lanes leave
// together with the same result also when the barrier completes around the last
// try (warp-wide instructions follow on both ways).
__device__ __forceinline__ bool sl_wait_warp(uint64_t* bar, uint32_t parity, int tries) {
    for (int it = 0; it < tries; ++it)
        if (__all_sync(0xffffffffu, sl_try(bar, parity))) return true;
    return false;
}
// the block's abort flag, the same answer for a whole warp
__device__ __forceinline__ bool sl_abort(volatile int* flag) { return __any_sync(0xffffffffu, *flag); }
__device__ __forceinline__ void sl_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], "
        "%4;" ::"r"(sl_addr(dst)),
        "l"(src), "r"(bytes), "r"(sl_addr(bar)), "l"(pol)
        : "memory");
}
// One lane of a converged warp.  The MMA warp runs as a whole and issues under
// elect.sync, so that the operands stay in uniform registers.
__device__ __forceinline__ bool sl_elect() {
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void sl_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sl_addr(bar))
                 : "memory");
}
// D (+)= A B: A 128 x 16 FP16 in TMEM, B N x 16 FP16 in shared memory (K-major, 64B swizzle)
template <bool ACC>
__device__ __forceinline__ void sl_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "n"(ACC ? 1 : 0));
}
__device__ __forceinline__ void tmem_ld4(uint32_t t, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(t));
}

// exponent ex with |v| < 2^ex for the largest |v| of a vector, from its bit
// pattern (the patterns of non-negative doubles order like the values, NaN above
// infinity) and n, the sources that are summed: from -1073 (the smallest
// subnormal) to 1026, kSlNan when it is not finite
constexpr int kSlNan = 1 << 16;
__device__ __forceinline__ int sl_exp(unsigned long long mbits, int n) {
    if (mbits >= 0x7ff0000000000000ull) return kSlNan;
    const double m = __longlong_as_double((long long)mbits);
    const int spare = n <= kSlExact ? 0 : n <= 4 * kSlExact ? 1 : 2;
    return (m > 0.0 ? ilogb(m) + 1 : 0) + spare;
}
// 2^e for -1022 <= e <= 1023
__device__ __forceinline__ double sl_pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
__device__ __forceinline__ double sl_nan() { return __longlong_as_double(0x7ff8000000000000ll); }
// Bytes d_t + 128 of the digits of rn(v 2^(54 - ex)), least significant first:
// balanced digits are the bytes of I + sum_t 128 256^t.  From the bit pattern:
// FP64 conversions run at the FP64 rate.
__device__ __forceinline__ unsigned long long sl_digits(double v, int ex) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(b >> 52) & 0x7ff;
    unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
    // v = +-m 2^(max(e, 1) - 1075) below 2^ex: a shift to the left (by at most one,
    // more only for subnormal v) stays below 2^54
    const int sh = max(e, 1) - 1021 - ex;
    m = sh < -54 ? 0ull : sh >= 0 ? m << min(sh, 63) : (m + (1ull << (-sh - 1))) >> -sh;
    return ((long long)b < 0 ? 0ull - m : m) + 0x80808080808080ull;
}
__device__ __forceinline__ unsigned long long sl_abs(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// FP16 digits of weight 256^-t of 8 numbers
__device__ __forceinline__ uint4 sl_halves(const unsigned long long (&d)[8], int t) {
    const int by = kSl - 1 - t;
    const __half2 off = __floats2half2_rn(1152.f, 1152.f);
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        // FP16 0x6400 | byte = 1024 + byte; minus 1152 gives the digit
        const uint32_t p = by < 4 ? __byte_perm((uint32_t)d[2 * q], (uint32_t)d[2 * q + 1], by | (4 + by) << 4)
                                  : __byte_perm((uint32_t)(d[2 * q] >> 32), (uint32_t)(d[2 * q + 1] >> 32), (by - 4) | by << 4);
        const uint32_t f = __byte_perm(p, 0x64646464u, 0x4140);
        const __half2 x = __hsub2(*reinterpret_cast<const __half2*>(&f), off);
        w[q] = *reinterpret_cast<const uint32_t*>(&x);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace
}  // namespace emsurf
