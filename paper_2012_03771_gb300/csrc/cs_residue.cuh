// K mod p for primes 2^28 <= p < 2^40 from K's 32-bit limbs.
//
// Exact division by 2^32 (K. Hensel; Montgomery's REDC of a long number): with
// s = 0, for each limb k_i from the lowest, s <- (s + k_i + m p) / 2^32, where m
// makes the sum divisible.  After n limbs s = K 2^(-32 n) (mod p): a limb costs
// three multiplies (two for p < 2^32), against the two full 64-bit products per
// 64-bit word of a Montgomery product over K's factors.  2^(32 n) is put back by
// one product with 2^(32 n + 64) mod p, which takes a power of two near 2 n + 64
// from float quotients and four squarings.
#pragma once
#include <stdint.h>

#include "cs_arith.cuh"

namespace cs {

// P32: 2^28 <= p < 2^32, else 2^32 < p < 2^40 (launch_res picks the form by the chunk,
// which does not cross 2^32).  ninv = -p^-1 mod 2^32.
struct ResMod {
    uint64_t p;
    uint32_t p0, p1, ninv;
    float rp;                   // 2^res_shift / p
};
// dropped low bits of a number whose quotient by p is estimated: |x| < 2^62 (P32:
// 2^54) keeps 31 bits, and the dropped part is below p / 2 (p >= 2^32; P32: 2^28)
template <bool P32>
CS_HD constexpr int res_shift() { return P32 ? 24 : 31; }
template <bool P32>
CS_HD ResMod res_mod(uint64_t p) {
    ResMod m;
    m.p = p;
    m.p0 = (uint32_t)p;
    m.p1 = P32 ? 0u : (uint32_t)(p >> 32);
    m.ninv = mont32_neg_inv(m.p0);
    m.rp = rcp_rn(u64_to_f(p)) * (P32 ? 16777216.0f : 2147483648.0f);
    return m;
}

// (t + m p) / 2^32 for the m < 2^32 that makes it whole; t < 2^52, the result at
// most t / 2^32 + p.  (t's low word plus m p0's is 0 mod 2^32, and m p0 + that word
// is below 2^64.)
template <bool P32>
CS_HD uint64_t res_step(uint64_t t, const ResMod &q) {
    const uint32_t m = (uint32_t)t * q.ninv;
    const uint64_t u = (uint64_t)m * q.p0 + (uint32_t)t;
    uint64_t s = (t >> 32) + (u >> 32);
    if (!P32) s += (uint64_t)m * q.p1;
    return s;
}

// One step of the chain on t = s + k_i: (t + m p) / 2^32 + k_(i+1), the quotient in
// [0, p + 1].  The low product takes the whole of t as its addend, which needs
// (2^32 - 1) p0 + t < 2^64: p0 <= 2^32 - 5 for P32 (the largest prime of 32 bits;
// t < 2^33), else p0 <= RES_P0_MAX (t < 2^41 + 2^32).
constexpr uint32_t RES_P0_MAX = 0xfffff7ffu;
template <bool P32>
CS_HD uint64_t res_limb(uint64_t t, uint32_t next, const ResMod &q) {
    const uint32_t m = (uint32_t)t * q.ninv;
    const uint32_t h = (uint32_t)(((uint64_t)m * q.p0 + t) >> 32);
    return P32 ? (uint64_t)h + next : (uint64_t)m * q.p1 + h + next;
}

// a b 2^-64 mod p, below p + 2^20, for a, b < 2^41.  In two words: (a0 b + m p) /
// 2^32 <= 2^41 + p, plus a1 b < 2^50 before the second step.  P32: at most p + 1, for
// a, b <= p + 1 (below 2^32): (a b + m p) / 2^32 < 2^33, and (2^33 + m p) / 2^32 < p + 2.
template <bool P32>
CS_HD uint64_t res_mul(uint64_t a, uint64_t b, const ResMod &q) {
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), b0 = (uint32_t)b, b1 = (uint32_t)(b >> 32);
    const uint64_t x = (uint64_t)a0 * b0;
    if (P32) {
        const uint64_t t = (x >> 32) + (((uint64_t)((uint32_t)x * q.ninv) * q.p0 + (uint32_t)x) >> 32);
        return ((uint64_t)((uint32_t)t * q.ninv) * q.p0 + t) >> 32;
    }
    const uint32_t m = (uint32_t)x * q.ninv;
    const uint64_t u = (uint64_t)m * q.p0 + (uint32_t)x;
    uint64_t t = (x >> 32) + (u >> 32) + (uint64_t)a0 * b1 + (uint64_t)a1 * b0 + ((uint64_t)(a1 * b1) << 32);
    if (!P32) t += (uint64_t)m * q.p1;
    return res_step<P32>(t, q);
}

// x - k p for an integer k near x / p, |x / p| < 2.5 2^20: the quotient of the
// upper bits in float (within 2^-22 of itself, below it by the dropped bits), made
// an integer by adding 1.5 2^23.  The result is in (-1.1 p, 1.7 p); for |x / p| <
// 1.5 2^20 in (-0.9 p, 1.4 p).
template <bool P32>
CS_HD int64_t res_near(int64_t x, const ResMod &q) {
    const float f = (float)(int32_t)(x >> res_shift<P32>());
#if defined(__CUDA_ARCH__)
    const int32_t k = (int32_t)((uint32_t)__float_as_int(__fmaf_rn(f, q.rp, 12582912.0f)) - 0x4B400000u);
#else
    const int32_t k = (int32_t)lrintf(f * q.rp);
#endif
    return x - (int64_t)k * (int64_t)q.p;
}

// 2^e mod p up to a multiple of p, in [0, 1.4 p) (P32: below p), for e >= 39: 2^20 ..
// 2^39, then 2^20 at a time
template <bool P32>
CS_HD uint64_t res_pow2(uint32_t e, const ResMod &q) {
    uint32_t done = 20 + e % 20;
    int64_t x = res_near<P32>((int64_t)1 << done, q);
    for (; done < e; done += 20) x = res_near<P32>((int64_t)((uint64_t)x << 20), q);
    if (x < 0) x += (int64_t)q.p;
    return (uint64_t)(P32 && x >= (int64_t)q.p ? x - (int64_t)q.p : x);
}

// 2^(32 n + 64) mod p up to a multiple of p (below p + 2^20): with the product's
// 2^-64, squaring takes 2^(64 + d) to 2^(64 + 2 d), so four squarings take
// 2^(64 + 2 n) there (a squaring costs as much as three steps of 2^20).
template <bool P32>
CS_HD uint64_t res_back(uint32_t n, const ResMod &q) {
    uint64_t y = res_pow2<P32>(2 * n + 64, q);
#pragma unroll
    for (int k = 0; k < 4; k++) y = res_mul<P32>(y, y, q);
    return y;
}

// the chain's end times 2^(32 n), reduced
template <bool P32>
CS_HD uint64_t res_finish(uint64_t s, uint32_t n, const ResMod &q) {
    const uint64_t r = res_mul<P32>(s, res_back<P32>(n, q), q);
    return r >= q.p ? r - q.p : r;
}

// (r M + s) mod p for r < p, M < 2^40, s < 2^20: r times the upper and the lower
// 20 bits of M, each reduced by one float quotient.
template <bool P32>
CS_HD uint64_t res_affine(uint64_t r, uint64_t M, uint32_t s, const ResMod &q) {
    int64_t x = 0;
    if (M >> 20) x = res_near<P32>((int64_t)(r * (M >> 20)), q);
    x = res_near<P32>((int64_t)(((uint64_t)x << 20) + r * (M & 0xfffffu)), q) + (int64_t)s;
    if (x < 0) x += (int64_t)q.p;
    if (x < 0) x += (int64_t)q.p;
    if (x >= (int64_t)q.p) x -= (int64_t)q.p;
    return x >= (int64_t)q.p ? (uint64_t)x - q.p : (uint64_t)x;
}

// x - k p for the integer k nearest to the float quotient, any p < 2^40, |x / p| <
// 2.5 2^20, |x| < 2^62 (rp within 2^-22 of 1 / p): the quotient is off by less than
// 1.4, so the result is within 1.5 p.
CS_HD int64_t near_rem(int64_t x, uint64_t p, float rp) {
#if defined(__CUDA_ARCH__)
    const float f = __fmaf_rn((float)(int32_t)(x >> 32), 4294967296.0f, (float)(uint32_t)x);
    const int32_t k = __float2int_rn(f * rp);
#else
    const float f = (float)(int32_t)(x >> 32) * 4294967296.0f + (float)(uint32_t)x;
    const int32_t k = (int32_t)lrintf(f * rp);
#endif
    return x - (int64_t)k * (int64_t)p;
}
// (r M + s) mod p for r < p < 2^40, M < 2^40, s <= p, as res_affine
CS_HD uint64_t near_affine(uint64_t r, uint64_t M, uint32_t s, uint64_t p) {
    const float rp = rcp_rn(u64_to_f(p));
    int64_t x = 0;
    if (M >> 20) x = near_rem((int64_t)(r * (M >> 20)), p, rp);
    if (x < 0) x += (int64_t)p;              // so that the halves of the next float do not cancel
    x = near_rem((int64_t)(((uint64_t)x << 20) + r * (M & 0xfffffu)), p, rp) + (int64_t)s;
    if (x < 0) x += (int64_t)p;
    if (x < 0) x += (int64_t)p;
    if (x >= (int64_t)p) x -= (int64_t)p;
    if (x >= (int64_t)p) x -= (int64_t)p;
    return (uint64_t)x;
}

// x 2^32 / p within 2, modulo 2^32, for x < p < 2^40: 16 bits of the
// quotient at a time
CS_HD uint32_t near_frac32(uint64_t x, uint64_t p, float rp) {
    int32_t k1 = (int32_t)(u64_to_f(x) * 65536.0f * rp);
    int64_t r1 = (int64_t)((x << 16) - (uint64_t)k1 * p);
    if (r1 < 0) {
        r1 += (int64_t)p;
        k1--;
    }
    const int32_t k2 = (int32_t)(u64_to_f((uint64_t)r1) * 65536.0f * rp);
    return ((uint32_t)k1 << 16) + (uint32_t)k2;
}

}  // namespace cs
