// Device helpers shared by the sampling kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mcpd {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of the 4x32 S-box with the Weyl
// key schedule.
static __device__ __forceinline__ uint4 philox10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        if (round) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// The same with the round keys (k0 + i W0, k1 + i W1), i = 0..9, given as rk[2 i], rk[2 i + 1].
static __device__ __forceinline__ uint4 philox10_rk(uint4 c, const uint32_t (&rk)[20]) {
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ rk[2 * round], lo1, hi0 ^ c.w ^ rk[2 * round + 1], lo0);
    }
    return c;
}

constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u, kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;

// Rounds 3 to 10 on the state after two rounds: with the third round's keys, or the key table above.
static __device__ __forceinline__ uint4 philox_tail(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int round = 2; round < 10; ++round) {
        if (round > 2) { k0 += kPhiloxW0; k1 += kPhiloxW1; }
        const uint32_t hi0 = __umulhi(kPhiloxM0, c.x), lo0 = kPhiloxM0 * c.x;
        const uint32_t hi1 = __umulhi(kPhiloxM1, c.z), lo1 = kPhiloxM1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}
static __device__ __forceinline__ uint4 philox_tail_rk(uint4 c, const uint32_t (&rk)[20]) {
#pragma unroll
    for (int round = 2; round < 10; ++round) {
        const uint32_t hi0 = __umulhi(kPhiloxM0, c.x), lo0 = kPhiloxM0 * c.x;
        const uint32_t hi1 = __umulhi(kPhiloxM1, c.z), lo1 = kPhiloxM1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ rk[2 * round], lo1, hi0 ^ c.w ^ rk[2 * round + 1], lo0);
    }
    return c;
}

// Word 0 of a block, out of line (the rare draw of a uniform's low half).
static __device__ __noinline__ uint32_t philox_low_word(uint4 c, uint32_t k0, uint32_t k1) {
    return philox10(c, k0, k1).x;
}

// Fire-and-forget global reductions (no value returned, no wait).
static __device__ __forceinline__ void red_add(long long *a, long long v) {
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}
static __device__ __forceinline__ void red_or(uint32_t *a, uint32_t v) {
    asm volatile("red.global.or.b32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}
static __device__ __forceinline__ void red_max(unsigned long long *a, unsigned long long v) {
    asm volatile("red.global.max.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}
// W(u) for any lag: sum_{r=k}^{min(l,u)} (floor((u - r) / lag) + 1) = (m - k + 1) + F(u - k) - F(u - m - 1),
// m = min(u, l), F(n) = sum_{d=0}^{n} floor(d / lag) = lag q (q - 1) / 2 + q (n - q lag + 1) with
// q = floor(n / lag).  32-bit divisions (every argument is a step count; with 64-bit ones a pair with
// lag one sweep spent most of its steps in them), and one of them only beyond l.
static __device__ __noinline__ long long lag_prefix(uint32_t u, uint32_t k, uint32_t ell, uint32_t lag) {
    if (u < k) return 0;
    const uint32_t m = min(u, ell);
    auto F = [&](uint32_t n) -> long long {
        const uint32_t q = n / lag;
        const unsigned long long lq = static_cast<unsigned long long>(lag) * q;
        return static_cast<long long>(q ? lq * (q - 1u) / 2u + static_cast<unsigned long long>(q) * (n - lq + 1u) : 0ull);
    };
    return static_cast<long long>(m - k + 1u) + F(u - k) - (u > m ? F(u - m - 1u) : 0ll);
}

// Add s1 and the 128-bit s2 = (lo, hi), carried into the high word, to clone j of bucket bkt.
static __device__ __forceinline__ void bucket_add_sums(unsigned long long *S1, unsigned long long *S2lo,
                                                unsigned long long *S2hi, int na, int bkt, int j, long long s1,
                                                unsigned long long lo, unsigned long long hi) {
    const size_t idx = static_cast<size_t>(bkt) * na + j;
    atomicAdd(&S1[idx], static_cast<unsigned long long>(s1));
    const unsigned long long old = atomicAdd(&S2lo[idx], lo);
    const unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
    if (hi + carry) atomicAdd(&S2hi[idx], hi + carry);
}
// Add G and G^2 of one slot to bucket N*_p - 1; or in two parts, the second with what the first returned.
static __device__ __forceinline__ void bucket_add(unsigned long long *S1, unsigned long long *S2lo,
                                           unsigned long long *S2hi, int na, int bkt, int j, long long g) {
    const unsigned long long a = static_cast<unsigned long long>(g < 0 ? -g : g);
    bucket_add_sums(S1, S2lo, S2hi, na, bkt, j, g, a * a, __umul64hi(a, a));
}
static __device__ __forceinline__ unsigned long long bucket_add_low(unsigned long long *S1, unsigned long long *S2lo,
                                                             int na, int bkt, int j, long long g) {
    const size_t idx = static_cast<size_t>(bkt) * na + j;
    atomicAdd(&S1[idx], static_cast<unsigned long long>(g));
    return atomicAdd(&S2lo[idx], static_cast<unsigned long long>(g) * static_cast<unsigned long long>(g));
}
static __device__ __forceinline__ void bucket_add_high(unsigned long long *S2hi, int na, int bkt, int j, long long g,
                                                unsigned long long old) {
    const unsigned long long a = static_cast<unsigned long long>(g < 0 ? -g : g), lo = a * a;
    const unsigned long long hi = __umul64hi(a, a) + (old + lo < old ? 1ull : 0ull);
    if (hi) atomicAdd(&S2hi[static_cast<size_t>(bkt) * na + j], hi);
}

}  // namespace mcpd
