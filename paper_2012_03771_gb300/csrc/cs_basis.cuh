// The three-gap walk's two steps and first hit in short chains: nearest-integer
// Euclid steps on float quotients, and a first hit found next to the walk's
// start in the basis of the two steps.
//
// Both rest on lattice facts that do not need exact quotients.  L = {(m, y) :
// y = r m (mod p)} has determinant p.
//
// * near_steps.  Every step x_(k+1) = x_(k-1) - q x_k, m_(k+1) = m_(k-1) - q m_k
//   with an integer q keeps (m_(k-1), x_(k-1)), (m_k, x_k) a basis of L, so q may
//   be any integer near the quotient; the nearest one halves |x| at least and
//   takes about 30% fewer steps than the floor (Hurwitz's nearest-integer
//   continued fraction).  The steps run until |x_k| <= w.  The walk's two steps
//   (a, -da) and (b, ub) are the only basis of L with a, b > 0, 1 <= da, ub <= w
//   and da + ub > w (a vector i (a, -da) + j (b, ub) with 0 < |y| <= w and m > 0
//   has i, j >= 0, so a and b are the smallest m of either sign): one of them is
//   the last vector found, the other the vector before it moved by t times the
//   last one until its y is in (w - d, w].  What is returned has been checked
//   against that description, so it is right whatever the quotients were.
//   64-bit p: the first steps are 64-bit ones, until the remainders fit 32 bits
//   (running them on leading digits with one 64-bit product at the end, after D.
//   H. Lehmer, measured 26 ps per prime against 15).
// * near_first_hit.  The lattice point next to (0, y = 0) of the walk's shifted
//   lattice comes from v0 a / p and v0 b / p in float; what is left to the first
//   hit is a few cells of the basis, in 32-bit arithmetic.
//
// Each returns false when its operands are outside the range its comments
// derive (rare: a tiny last remainder, a start inside a long run of one step);
// the caller then takes the general routines of cs_arith.cuh, whose answers are
// the same.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "cs_arith.cuh"

namespace cs {

// rint(x) for |x| < 2^22 by adding 1.5 2^23: the sum's low mantissa bits are the
// integer (round to nearest), and subtracting it again gives it as a float.
constexpr float NEAR_MAGIC = 12582912.0f;
CS_HD int32_t float_bits(float x) {
#if defined(__CUDA_ARCH__)
    return __float_as_int(x);
#else
    int32_t i;
    memcpy(&i, &x, 4);
    return i;
#endif
}
CS_HD float near_fma(float a, float b, float c) {
#if defined(__CUDA_ARCH__)
    return __fmaf_rn(a, b, c);
#else
    return fmaf(a, b, c);
#endif
}
CS_HD int32_t near_int(float sum) { return (int32_t)((uint32_t)float_bits(sum) - 0x4B400000u); }

// float of a signed 64-bit number through its halves: within 2^8 + 2^-22 |x|
CS_HD float near_s64_to_f(int64_t x) {
    return near_fma((float)(int32_t)(x >> 32), 4294967296.0f, (float)(uint32_t)x);
}
CS_HD int32_t near_abs(int32_t x) { return x < 0 ? -x : x; }

// ceil(n / d) for |n| < 2^31, 1 <= d < 2^31 and |n / d| < 2^20, rd within a
// relative 2^-22 of 1 / d: the float quotient is within 1/2 + 2^20 2^-21 of n / d
// before its rounding up, so it is the ceiling or off by one either way.
CS_HD int32_t near_ceil_div(int32_t n, int32_t d, float rd) {
    int32_t q = (int32_t)ceilf((float)n * rd);
    const int32_t r = q * d - n;                 // wanted in [0, d)
    if (r < 0) q++;
    else if (r >= d) q--;
    return q;
}

// The steps (a, -da), (b, ub) of 0 < r < p, gcd(r, p) = 1, and a window w with
// 512 <= w <= 2^21, p < 2^30 (UT = uint32_t) or p < 2^40, p < 2^28 w and w >= 1024
// (UT = uint64_t).  From the determinant |m_k x_(k-1) - m_(k-1) x_k| = p and
// |x_k| <= |x_(k-1)| / 2 or little more, |m_k| <= 4 p / |x_(k-1)| also with a
// quotient that is off (the last 64-bit one, of a remainder that its upper bits
// hardly show), so every m taken while |x_(k-1)| > w is below 4 p / w <= 2^30.
// False: outside these bounds, or a quotient beyond 2^21.
template <class UT>
CS_HD bool near_steps(UT p, UT r, uint32_t w, uint32_t &a, uint32_t &da, uint32_t &b, uint32_t &ub,
                      uint32_t &iters) {
    int32_t x0, x1, m0, m1;
    uint32_t k = 0;
    const int32_t wi = (int32_t)w;
    if (sizeof(UT) == 8) {
        // 64-bit steps, their quotients from the values' upper 30 bits, until both
        // are below 2^31 (a mean of two steps at p = 5e10)
        if ((uint64_t)p >> 28 >= w) return false;
        int64_t y0 = (int64_t)p, y1 = (int64_t)r;
        int32_t n0 = 0, n1 = 1;
        float g0 = (float)(int32_t)(y0 >> 10);
        bool more = true;
        do {
            const float g1 = (float)(int32_t)(y1 >> 10);
            const float qf = g0 * rcp_approx(g1);
            if (!(fabsf(qf) < 2097152.0f)) return false;
            const int32_t q = near_int(near_fma(qf, 1.0f, NEAR_MAGIC));
            const int64_t y2 = y0 - (int64_t)q * y1;
            const int32_t n2 = (int32_t)((uint32_t)n0 - (uint32_t)q * (uint32_t)n1);
            more = (uint64_t)(y1 + 0x40000000) > 0x80000000ull && k < 32;
            y0 = y1; n0 = n1; g0 = g1;
            y1 = y2; n1 = n2;
            k++;
        } while (more);
        if (k >= 32 || y1 != (int64_t)(int32_t)y1 || (y0 >= -(int64_t)wi && y0 <= (int64_t)wi)) return false;
        x0 = (int32_t)y0; x1 = (int32_t)y1;
        m0 = n0; m1 = n1;
    } else {
        x0 = (int32_t)p; x1 = (int32_t)r;
        m0 = 0; m1 = 1;
    }
    // 32-bit steps, two a pass, until the last one is in the window
    float f0 = (float)x0, f1 = (float)x1;
    if ((uint32_t)(x1 + wi) > 2 * w) {               // |x1| > w
        for (;;) {
            int32_t q = near_int(near_fma(f0, rcp_approx(f1), NEAR_MAGIC));
            x0 = (int32_t)((uint32_t)x0 - (uint32_t)q * (uint32_t)x1);
            m0 = (int32_t)((uint32_t)m0 - (uint32_t)q * (uint32_t)m1);
            f0 = (float)x0;
            k++;
            if ((uint32_t)(x0 + wi) <= 2 * w) {
                const int32_t x = x0, m = m0;
                x0 = x1; m0 = m1; x1 = x; m1 = m;
                break;
            }
            q = near_int(near_fma(f1, rcp_approx(f0), NEAR_MAGIC));
            x1 = (int32_t)((uint32_t)x1 - (uint32_t)q * (uint32_t)x0);
            m1 = (int32_t)((uint32_t)m1 - (uint32_t)q * (uint32_t)m0);
            f1 = (float)x1;
            k++;
            if ((uint32_t)(x1 + wi) <= 2 * w || k > 96) break;
        }
        if (k > 96) return false;
    }
    iters += k;
    // the last vector with m > 0; y reflected where needed so that its y is -d
    const bool flip = m1 < 0;
    if (flip) { m1 = -m1; x1 = -x1; }
    const bool down = x1 < 0;
    const int32_t d = down ? -x1 : x1;
    int32_t u = down ? x0 : -x0;
    // the vector before it, oriented: m1 u + m0 d = +p (mod 2^32 tells +p from -p)
    const uint32_t det = (uint32_t)m1 * (uint32_t)u + (uint32_t)m0 * (uint32_t)d;
    if (det != (uint32_t)p) { m0 = -m0; u = -u; }
    // t = ceil((u - w) / d) puts its y into (w - d, w]
    const float rd = rcp_approx((float)d);
    const float tf = (float)(u - wi) * rd;
    // |x0| <= 2^30 (the subtraction above is exact), the quotient below 2^20, and b = m0 + t m1 below 2^30
    if (d == 0 || m1 == 0 || near_abs(x0) > (1 << 30) || !(fabsf(tf) < 1048576.0f) ||
        !(fabsf(tf) * (float)m1 + fabsf((float)m0) < 1.07e9f) || m1 > (1 << 30))
        return false;
    const int32_t t = near_ceil_div(u - wi, d, rd);
    const int32_t v = u - t * d, mb = m0 + t * m1;
    if (mb <= 0 || v <= 0 || v > wi || v + d <= wi) return false;
    // the determinant: m1 v + mb d = p
    if ((uint64_t)(uint32_t)m1 * (uint32_t)v + (uint64_t)(uint32_t)mb * (uint32_t)d != (uint64_t)p) return false;
    a = (uint32_t)(down ? m1 : mb); da = (uint32_t)(down ? d : v);
    b = (uint32_t)(down ? mb : m1); ub = (uint32_t)(down ? v : d);
    return true;
}

// The smallest t >= 0 with (v0 + r t) mod p <= w, and that residue, from the
// two steps of r (p < 2^40, w <= 2^21), for w < v0 < p; fp = a float within a
// relative 2^-22 of p's reciprocal.
//
// As in first_hit32 the strip is reflected so that the finer step DA = min(da,
// ub) leads down: block j holds the points (t, y) = i (A, -DA) + j (B, UB) of one
// j, and the answer is the first point with t >= 0 of the first block that has
// one.  A UB + B DA = p, and the point i0 = V0 B / p, j0 = -V0 A / p (rounded
// from float, off by 1/2 + 2^-21 B and 1/2 + 2^-21 A) lies at y0, t0 with
//   |y0| <= w + p 2^-20 < 2^23 and |t0| <= (A + B) / 2 + A B 2^-20,
// both small enough to be taken modulo 2^32.  From there the first block is
// ceil(-(t0 DA + y0 A) / p) or one of the next two; the sizes that follow from
// that are checked before the blocks are tried.
CS_HD bool near_first_hit(float fp, uint32_t w, uint32_t a, uint32_t da, uint32_t b, uint32_t ub, uint64_t v0,
                          uint32_t &t_out, uint32_t &y_out) {
    const bool sw = da > ub;
    const uint32_t A = sw ? b : a, DA = sw ? ub : da, B = sw ? a : b, UB = sw ? da : ub;
    const float fA = (float)A, fB = (float)B, fD = (float)DA, fw = (float)w;
    // V0 = v0, or the reflected start w - v0
    const int64_t V0 = sw ? (int64_t)w - (int64_t)v0 : (int64_t)v0;
    const float f = near_s64_to_f(V0) * fp;
    const int32_t i0 = (int32_t)rintf(f * fB), j0 = -(int32_t)rintf(f * fA);
    const int32_t t0 = (int32_t)((uint32_t)i0 * A + (uint32_t)j0 * B);
    const int32_t y0 = (int32_t)((uint32_t)V0 - (uint32_t)i0 * DA + (uint32_t)j0 * UB);
    // first block, taken a little low: the loop moves up
    const float ft = (float)t0, fy = (float)y0;
    const float jr = -(ft * fD + fy * fA) * fp;
    int32_t j = (int32_t)ceilf(jr - 9.765625e-4f);
    // over the blocks tried, |T| < bt < 2^31 with quotients by A below 2^20, and
    // |Y - w| < by with quotients by DA below 2^20 (t0's own bound: bt covers it)
    const float bj = fabsf(jr) + 6.0f, bt = bj * fB + fA + fA * fB * 1.0e-6f, by = bj * fw + fabsf(fy);
    if (!(bt < 2.1e9f) || !(bt < fA * 1048576.0f) || !(by < fD * 1048576.0f)) return false;
    const float rA = rcp_approx(fA), rD = rcp_approx(fD);
    for (int n = 0; n < 5; n++, j++) {
        const int32_t Y = y0 + j * (int32_t)UB, T = t0 + j * (int32_t)B;
        const int32_t iy = near_ceil_div(Y - (int32_t)w, (int32_t)DA, rD);   // y <= w from here on
        const int32_t it = near_ceil_div(-T, (int32_t)A, rA);                // t >= 0 from here on
        const int32_t i = iy > it ? iy : it;
        const int32_t y = Y - i * (int32_t)DA;
        if (y >= 0) {
            t_out = (uint32_t)(T + i * (int32_t)A);
            y_out = sw ? w - (uint32_t)y : (uint32_t)y;
            return true;
        }
    }
    return false;
}

}  // namespace cs
