// Sieving-prime source: a segmented sieve of Eratosthenes over odd numbers,
// fused with the cached residue r = K mod p of Section 3.1 (Space-Time
// Tradeoff).  The paper treats prime generation up to P_limit as a small
// one-time cost (Runtime section); here it runs on the device so that the
// primes never cross the host boundary.
//
// One CTA sieves one segment of SEG odd numbers in shared memory at a time
// (grid-stride over segments).  The multiples of 3..31 come from tabulated
// period masks; those of the other base primes q <= sqrt(hi) are marked with
// shared-memory atomics: small q cooperatively by a warp, large q one per
// thread, their first multiples from float quotients.  The CTA takes the output
// entries of a whole segment with one atomic; each warp then scans its share of
// the segment, queues the primes it finds in shared memory and, 32 at a time,
// computes K mod p with Montgomery multiplication over K's prime factors packed
// into machine words (64-bit primes: the residue kernel after the sieve) and
// writes the entries.
//
// Bound: instruction issue.  Per prime near 9e9, about 16 marks (a shared-memory
// atomic and five instructions each), the first multiples of the base primes
// (twenty instructions each, per segment) and the extraction.
#include <atomic>

#include "cs_arith.cuh"
#include "cs_internal.h"
#include "cs_residue.cuh"

namespace cs {

namespace {

// base primes marked by a whole warp (below) or one thread each (above): a
// warp's lanes on multiples of one q >= 1024 fall on few shared-memory banks, one
// q per lane spreads them (1024 measured best of 128 to 16384)
constexpr uint32_t WARP_COOP_Q = 1024;
constexpr uint32_t N_COOP = 171;            // odd primes below it: the ascending base list reaches it there
// Every segment computes the first multiple of every base prime, whose number
// grows with sqrt(hi) (26,000 at 9e10), so segments are large: up to 2^18 odd
// numbers, two CTAs of 1024 threads per SM.  A list of the primes of 2^27 numbers
// at 9e8 / 9e9 / 9e10 takes 51 / 57 / 69 us (54 / 63 / 85 with four CTAs of 512
// threads, 61 / 76 / 107 with five of 256 and 2^17 odd numbers).
constexpr int GEN_MIN_BLOCKS = 2;
constexpr uint32_t SEG = 1u << 18;
constexpr uint32_t SEG_MIN = 1u << 10;      // smallest segment: 32 words
constexpr uint32_t SEG_WORDS = SEG / 32;
constexpr uint32_t GEN_THREADS = 1024;
constexpr uint32_t GEN_WARPS = GEN_THREADS / 32;
// per-warp queue: the primes of one step (32 words, 2048 consecutive numbers: at
// most 2 * 2048 / log 2048 = 537 by Montgomery and Vaughan) and 31 left over; kept
// as 16-bit positions in the warp's part of the segment
constexpr uint32_t QCAP = 576;
static_assert(SEG / GEN_WARPS <= 65536, "16-bit positions");
static_assert(SEG_MIN % (32 * GEN_WARPS) == 0, "whole words per warp");

// SMALL: tile records; LARGE32: (p, r, v0) of one plan; LIST: 64-bit p only (the
// residue kernel adds r and v0 for a plan, r for a cache); PR32: (p, r) for a
// residue cache shared by plans with the same K
enum Kind { KIND_SMALL = 0, KIND_LARGE32 = 1, KIND_LIST = 2, KIND_PR32 = 3 };

struct GenArgs {
    uint64_t i_begin, i_end;      // odd indices [i_begin, i_end): numbers 2i+1
    uint64_t n_seg;
    uint32_t seg;                 // odd numbers per segment (multiple of SEG_MIN, <= SEG)
    bool emit_two;                // 2 is in range
    const uint32_t *base;         // odd base primes, ascending
    uint32_t n_base;
    // residue parameters
    const uint32_t *kch32;
    uint32_t n_kch32;
    const uint32_t *klimb;
    uint32_t n_klimb;
    uint64_t M_start;
    uint32_t SL;
    // outputs
    void *o0, *o1, *o2;
    uint64_t cap;
    unsigned long long *count;
    unsigned long long *err;
};

__device__ __forceinline__ uint32_t kmodp32(uint32_t p, uint32_t pinv, uint32_t r1, uint32_t r2,
                                            const uint32_t *kch, uint32_t n) {
    if (n == 0) return 1u % p;
    uint32_t acc = mont32_rpow(n, r1, r2, p, pinv);     // R^n: cancels the n factors R^-1
    // the factor words are below 2^31, so the running product stays below 2p;
    // four words per 16-byte load when the word array is aligned
    uint32_t i = 0;
    if ((reinterpret_cast<uintptr_t>(kch) & 15) == 0) {
        const uint4 *k4 = reinterpret_cast<const uint4 *>(kch);
        for (; i + 4 <= n; i += 4) {
            const uint4 w = __ldg(&k4[i / 4]);
            acc = mont32_mul_lazy(acc, w.x, p, pinv);
            acc = mont32_mul_lazy(acc, w.y, p, pinv);
            acc = mont32_mul_lazy(acc, w.z, p, pinv);
            acc = mont32_mul_lazy(acc, w.w, p, pinv);
        }
    }
    for (; i < n; i++) acc = mont32_mul_lazy(acc, __ldg(&kch[i]), p, pinv);
    return acc >= p ? acc - p : acc;
}

// slot: the output entry of this lane's prime
template <int KIND>
__device__ __forceinline__ void emit(const GenArgs &a, uint64_t p, bool valid, uint64_t slot) {
    // residue work for this lane's prime
    uint32_t e0 = 0, e1 = 0, e2 = 0, e3 = 0;
    uint64_t w0 = 0;
    if (valid) {
        if (KIND == KIND_SMALL) {
            uint32_t p32 = (uint32_t)p;
            if (p32 == 2) {
                // only when P < 2, so K = 1 and r = 1
                e0 = 2; e1 = 0; e2 = 1; e3 = (uint32_t)((a.M_start + a.SL) & 1);
            } else {
                uint32_t pinv = mont32_neg_inv(p32);
                uint32_t r1 = mont32_r1(p32), r2 = mont32_r2(p32);
                uint32_t r = kmodp32(p32, pinv, r1, r2, a.kch32, a.n_kch32);
                uint32_t rt = mont32_mul(r, r2, p32, pinv);
                uint32_t ms = (uint32_t)(a.M_start % p32);
                uint32_t v = mont32_mul(rt, ms, p32, pinv) + a.SL % p32;
                e0 = p32; e1 = pinv; e2 = rt; e3 = v >= p32 ? v - p32 : v;
            }
        } else if (KIND == KIND_LARGE32) {
            uint32_t p32 = (uint32_t)p;
            uint32_t pinv = mont32_neg_inv(p32);
            uint32_t r2 = mont32_r2_fast(p32);
            uint32_t r1 = mont32_mul(r2, 1u, p32, pinv);         // R mod p
            uint32_t r = kmodp32(p32, pinv, r1, r2, a.kch32, a.n_kch32);
            uint32_t rt = mont32_mul(r, r2, p32, pinv);
            e0 = p32; e1 = r; e2 = mont32_affine(rt, a.M_start, a.SL, r2, p32, pinv);   // SL < p
        } else if (KIND == KIND_PR32) {
            uint32_t p32 = (uint32_t)p;
            uint32_t pinv = mont32_neg_inv(p32);
            e0 = p32;
            const uint32_t r2 = mont32_r2_fast(p32);
            e1 = kmodp32(p32, pinv, mont32_mul(r2, 1u, p32, pinv), r2, a.kch32, a.n_kch32);
        } else {
            w0 = p;
        }
    }
    if (!valid) return;
    if (slot >= a.cap) {
        atomicOr(a.err, (unsigned long long)ERR_PRIME_OVERFLOW);
        return;
    }
    if (KIND == KIND_SMALL) {
        reinterpret_cast<SmallPrime *>(a.o0)[slot] = SmallPrime{e0, e1, e2, e3};
    } else if (KIND == KIND_LARGE32) {
        reinterpret_cast<uint32_t *>(a.o0)[slot] = e0;
        reinterpret_cast<uint32_t *>(a.o1)[slot] = e1;
        reinterpret_cast<uint32_t *>(a.o2)[slot] = e2;
    } else if (KIND == KIND_PR32) {
        reinterpret_cast<uint32_t *>(a.o0)[slot] = e0;
        reinterpret_cast<uint32_t *>(a.o1)[slot] = e1;
    } else {
        reinterpret_cast<uint64_t *>(a.o0)[slot] = w0;
    }
}

// Residues of the 64-bit primes the generator wrote (o0): r = K mod p (Section
// 3.1) into o1 and, for a plan, v = (r M_start + SL) mod p into o2.  RES_ILP
// primes per thread share the loads of K's limbs.  The 32-bit residues stay in
// the sieve kernel, where they fill issue slots that its barriers and marking
// phases leave idle.
//
// Bound: the wide multiplies (a 32 x 32 + 64-bit one takes a scheduler about
// five cycles, against one for an addition), two per limb and prime, one for p <
// 2^32.  K = 1019#/210 (44 limbs) at p = 5e10: 34 ps per prime (60 as 64-bit
// Montgomery products over 23 factor words), K = 1511#/210 (66 limbs) 43 (78), p <
// 2^32: 26 and 32.  One prime per thread: 40, three: 36 (44 limbs).
constexpr uint32_t RES_THREADS = 256;
constexpr int RES_ILP = 2;
template <bool P32>
__device__ __forceinline__ uint64_t res_k_mod_p(const ResMod &q, const uint32_t *limb, uint32_t n) {
    // a modulus whose low word is too near 2^32 for the chain's products
    if (q.p0 > RES_P0_MAX) {
        uint64_t s = 0;
        for (uint32_t i = 0; i < n; i++) s = res_step<P32>(s + __ldg(limb + i), q);
        return res_finish<P32>(s, n, q);
    }
    uint64_t t = __ldg(limb);
    for (uint32_t i = 1; i < n; i++) t = res_limb<P32>(t, __ldg(limb + i), q);
    return res_finish<P32>(res_limb<P32>(t, 0, q), n, q);
}
template <bool P32, bool V>
__global__ void __launch_bounds__(RES_THREADS) k_large_res(const GenArgs a) {
    const uint64_t n = min((uint64_t)*a.count, a.cap);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t *P = reinterpret_cast<const uint64_t *>(a.o0);
    const uint32_t nl = a.n_klimb;
    for (uint64_t i0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i0 < n; i0 += RES_ILP * stride) {
        ResMod q[RES_ILP];
        uint64_t t[RES_ILP];
        const uint32_t first = __ldg(a.klimb);
#pragma unroll
        for (int k = 0; k < RES_ILP; k++) {
            const uint64_t i = i0 + k * stride;
            q[k] = res_mod<P32>(i < n ? P[i] : P[i0]);       // the extra chains repeat a valid prime
            t[k] = first;
        }
#pragma unroll 4
        for (uint32_t l = 1; l < nl; l++) {
            const uint32_t w = __ldg(a.klimb + l);
#pragma unroll
            for (int k = 0; k < RES_ILP; k++) t[k] = res_limb<P32>(t[k], w, q[k]);
        }
#pragma unroll
        for (int k = 0; k < RES_ILP; k++) {
            const uint64_t i = i0 + k * stride;
            if (i >= n) continue;
            uint64_t r = res_finish<P32>(res_limb<P32>(t[k], 0, q[k]), nl, q[k]);
            if (!P32 && q[k].p0 > RES_P0_MAX) r = res_k_mod_p<false>(q[k], a.klimb, nl);
            reinterpret_cast<uint64_t *>(a.o1)[i] = r;
            if (V) reinterpret_cast<uint64_t *>(a.o2)[i] = res_affine<P32>(r, a.M_start, a.SL, q[k]);
        }
    }
}

// n mod q with 32-bit arithmetic when n fits (all segments below 2^32)
__device__ __forceinline__ uint32_t first_rem(uint64_t n, uint32_t q) {
    return (n >> 32) == 0 ? (uint32_t)n % q : (uint32_t)(n % q);
}

// Smallest k >= 0 with q | 2 (i0 + k) + 1, for odd 1024 <= q < 2^21 and i0 < 2^40
// (fi0 = i0 rounded to float): i0 + k = (q - 1)/2 (mod q).  i0 mod q from two float
// quotients without a 64-bit division: the first, i0 / q < 2^30, is off by less
// than 2^7 (three roundings of 2^-23 at most), so i0 less its multiple of q fits
// 32 signed bits and is taken modulo 2^32; the second, rounded, leaves a
// remainder within q/2 + 1 of 0.
__device__ __forceinline__ uint32_t first_multiple(uint64_t i0, float fi0, uint32_t q) {
    const float rq = rcp_approx((float)q);
    const uint32_t q1 = (uint32_t)(fi0 * rq);
    const int32_t r1 = (int32_t)((uint32_t)i0 - q1 * q);
    const int32_t q2 = __float2int_rn((float)r1 * rq);
    int32_t r = r1 - q2 * (int32_t)q;
    if (r < 0) r += (int32_t)q;
    int32_t k = (int32_t)(q >> 1) - r;
    if (k < 0) k += (int32_t)q;
    return (uint32_t)k;
}

// Pre-sieve of the odd multiples of 3..31 (half of all marks, and the ones
// whose lanes collide on the same shared-memory word): the masks of one period
// of T = 3*5*7, 11*13, 17*19, 23*29 and 31 odd indices are tabulated, and word w
// of a segment, whose first odd index I = i0 + 32 w has I mod T = s, ORs in table
// entry s.  Bit b of that entry is set when the odd number 2(I + b) + 1 has a
// factor q | T, i.e. I + b = (q - 1)/2 (mod q).  The tables are computed at
// compile time and copied to shared memory (computing them in every CTA cost
// about a seventh of a light chunk's generation).
constexpr int PRE_N = 5;
constexpr uint32_t PRE_MAX_Q = 31;
CS_HD constexpr uint32_t pre_T(int t) { return t == 0 ? 105 : t == 1 ? 143 : t == 2 ? 323 : t == 3 ? 667 : 31; }
CS_HD constexpr uint32_t pre_off(int t) {
    return t == 0 ? 0 : t == 1 ? 105 : t == 2 ? 248 : t == 3 ? 571 : t == 4 ? 1238 : 1269;
}
constexpr uint32_t PRE_WORDS = 1269;
struct PreTable {
    uint32_t w[PRE_WORDS];
};
constexpr PreTable make_pre_table() {
    PreTable t{};
    constexpr uint32_t qs[10] = {3, 5, 7, 11, 13, 17, 19, 23, 29, 31};
    for (int k = 0; k < PRE_N; k++)
        for (uint32_t s = 0; s < pre_T(k); s++) {
            uint32_t m = 0;
            for (int j = 0; j < 10; j++) {
                const uint32_t q = qs[j];
                if (pre_T(k) % q) continue;
                for (uint32_t b = ((q - 1) / 2 + q - s % q) % q; b < 32; b += q) m |= 1u << b;
            }
            t.w[pre_off(k) + s] = m;
        }
    return t;
}
__device__ const PreTable c_pre = make_pre_table();

template <int KIND>
__global__ void __launch_bounds__(GEN_THREADS, GEN_MIN_BLOCKS) k_gen(const GenArgs a) {
    extern __shared__ uint32_t gen_smem[];
    uint32_t *comp = gen_smem;                    // SEG_WORDS: bit set = composite (or out of range)
    uint32_t *pre = comp + SEG_WORDS;             // PRE_WORDS: pre-sieve tables
    uint16_t *queue = reinterpret_cast<uint16_t *>(pre + PRE_WORDS) + (threadIdx.x >> 5) * QCAP;
    __shared__ uint32_t warp_n[GEN_WARPS];        // primes in each warp's part of the segment
    __shared__ unsigned long long seg_base;       // output entry of the segment's first prime
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t e = threadIdx.x; e < PRE_WORDS; e += GEN_THREADS) pre[e] = c_pre.w[e];
    __syncthreads();

    if (a.emit_two && blockIdx.x == 0 && threadIdx.x == 0)
        emit<KIND>(a, 2, true, atomicAdd(a.count, 1ull));

    const uint32_t n_coop = min(N_COOP, a.n_base);   // base primes marked by whole warps

    for (uint64_t s = blockIdx.x; s < a.n_seg; s += gridDim.x) {
        const uint64_t i0 = a.i_begin + s * a.seg;
        const uint64_t i1 = min(i0 + a.seg, a.i_end);
        const uint32_t seg_words = a.seg / 32;
        const uint32_t len = (uint32_t)(i1 - i0);
        const uint64_t n_first = 2 * i0 + 1;
        const uint64_t n_last = 2 * (i1 - 1) + 1;
        // the tables apply when no q <= 31 lies in the segment itself
        const bool pre_ok = n_first > PRE_MAX_Q;
        uint32_t ph[PRE_N], step[PRE_N];
#pragma unroll
        for (int t = 0; t < PRE_N; t++) {
            const uint32_t T = pre_T(t);
            ph[t] = pre_ok ? first_rem(i0 + 32ull * threadIdx.x, T) : 0;
            step[t] = (32u * GEN_THREADS) % T;
        }
        for (uint32_t w = threadIdx.x; w < seg_words; w += GEN_THREADS) {
            uint32_t v = 0;
            uint32_t lo = w * 32;
            if (lo + 32 > len) v = lo >= len ? 0xffffffffu : (0xffffffffu << (len - lo));
            if (pre_ok) {
#pragma unroll
                for (int t = 0; t < PRE_N; t++) {
                    v |= pre[pre_off(t) + ph[t]];
                    ph[t] += step[t];
                    if (ph[t] >= pre_T(t)) ph[t] -= pre_T(t);
                }
            }
            comp[w] = v;
        }
        __syncthreads();
        if (i0 == 0 && threadIdx.x == 0) atomicOr(&comp[0], 1u);   // 1 is not prime

        // mark odd multiples of the base primes, starting at max(q^2, first in
        // segment).  Small ones by a whole warp each; its lanes compute the starts
        // of 32 of them at once
        for (uint32_t b0 = 0; b0 < n_coop; b0 += 32 * GEN_WARPS) {
            const uint32_t b = b0 + lane * GEN_WARPS + warp;
            uint32_t q_l = 0, k_l = 0xffffffffu;
            if (b < n_coop) {
                q_l = __ldg(&a.base[b]);
                const uint64_t sq = (uint64_t)q_l * q_l;
                if (sq <= n_last && !(pre_ok && q_l <= PRE_MAX_Q)) {
                    if (sq >= n_first) {
                        k_l = (uint32_t)((sq - n_first) >> 1);
                    } else {
                        const uint32_t r = first_rem(i0, q_l);
                        k_l = (q_l >> 1) >= r ? (q_l >> 1) - r : (q_l >> 1) + q_l - r;
                    }
                }
            }
            const uint32_t n_b = min(32u, (n_coop - b0 + GEN_WARPS - 1) / GEN_WARPS);
            for (uint32_t t = 0; t < n_b; t++) {
                const uint32_t q = __shfl_sync(0xffffffffu, q_l, t), k = __shfl_sync(0xffffffffu, k_l, t);
                if (k >= len) continue;
                for (uint32_t idx = k + lane * q; idx < len; idx += 32 * q)
                    atomicOr(&comp[idx >> 5], 1u << (idx & 31));
            }
        }
        // large base primes: one per thread (at most SEG / q + 1 marks each)
        {
            const float fi0 = (float)(uint32_t)(i0 >> 20) * 1048576.0f + (float)(uint32_t)(i0 & 0xfffffu);
            for (uint32_t b = n_coop + threadIdx.x; b < a.n_base; b += GEN_THREADS) {
                const uint32_t q = __ldg(&a.base[b]);
                const uint64_t sq = (uint64_t)q * q;
                if (sq > n_last) break;
                const uint64_t k = sq >= n_first ? (sq - n_first) >> 1 : first_multiple(i0, fi0, q);
                if (k >= len) continue;
                for (uint32_t idx = (uint32_t)k; idx < len; idx += q)
                    atomicOr(&comp[idx >> 5], 1u << (idx & 31));
            }
        }
        __syncthreads();

        // extract: each warp owns a contiguous run of words.  The segment's output
        // entries are taken with one atomic (one per 32 primes, all on the one
        // counter, stalled the warps on its latency)
        const uint32_t wpw = seg_words / GEN_WARPS;
        uint32_t cnt = 0;
        for (uint32_t w = warp * wpw + lane; w < (warp + 1) * wpw; w += 32) cnt += __popc(~comp[w]);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) warp_n[warp] = cnt;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t n = 0;
            for (uint32_t w = 0; w < GEN_WARPS; w++) n += warp_n[w];
            seg_base = n ? atomicAdd(a.count, (unsigned long long)n) : 0;
        }
        __syncthreads();
        uint64_t slot = seg_base;
        for (uint32_t w = 0; w < warp; w++) slot += warp_n[w];
        const uint64_t part = 2 * (i0 + (uint64_t)warp * wpw * 32) + 1;    // the part's first number
        uint32_t qlen = 0;
        for (uint32_t w0 = 0; w0 < wpw; w0 += 32) {
            const uint32_t w = w0 + lane;
            uint32_t primes = w < wpw ? ~comp[warp * wpw + w] : 0u;
            const uint32_t c = __popc(primes);
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (unsigned)o) incl += t;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            uint32_t pos = qlen + incl - c;
            while (primes) {
                queue[pos++] = (uint16_t)(w * 32 + __ffs(primes) - 1);
                primes &= primes - 1;
            }
            qlen += total;
            __syncwarp();
            uint32_t done = 0;
            while (qlen - done >= 32) {
                emit<KIND>(a, part + 2 * queue[done + lane], true, slot + lane);
                done += 32;
                slot += 32;
            }
            __syncwarp();
            // move the remainder (< 32 entries) to the front
            const uint32_t rest = qlen - done;
            const uint16_t keep = lane < rest ? queue[done + lane] : (uint16_t)0;
            __syncwarp();
            if (lane < rest) queue[lane] = keep;
            qlen = rest;
            __syncwarp();
        }
        if (lane < qlen) emit<KIND>(a, part + 2 * queue[lane], true, slot + lane);
        __syncthreads();
    }
}

constexpr size_t GEN_SMEM = (SEG_WORDS + PRE_WORDS) * 4 + GEN_WARPS * QCAP * 2;

// CTAs of k_gen<KIND> resident at once on the current device, whose shared-memory
// limit for the kernel is raised on the first call (once per kind and device)
template <int KIND>
int gen_resident() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    int n = cached[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        int per_sm = 0;
        cudaFuncSetAttribute(k_gen<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GEN_SMEM);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gen<KIND>, GEN_THREADS, GEN_SMEM) != cudaSuccess ||
            per_sm <= 0)
            per_sm = 1;
        n = sm_count() * per_sm;
        cached[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

GenArgs make_args(uint64_t lo, uint64_t hi, const uint32_t *base, uint32_t n_base, int resident) {
    GenArgs a{};
    a.base = base;
    a.n_base = n_base;
    if (hi <= lo || hi < 2) {
        a.n_seg = 0;
        return a;
    }
    a.i_begin = (lo + 1) / 2;
    a.i_end = (hi + 1) / 2;
    const uint64_t odds = a.i_end > a.i_begin ? a.i_end - a.i_begin : 0;
    uint32_t seg = SEG_MIN;
    // segment size: the range split evenly over whole waves of the resident
    // CTAs (k segments each), in multiples of SEG_MIN within [SEG_MIN, SEG], so
    // that no CTA waits on a partly filled last wave
    {
        const uint64_t res = (uint64_t)(resident > 0 ? resident : 1);
        const uint64_t k = (odds + res * SEG - 1) / (res * SEG);               // segments per CTA
        const uint64_t per = k ? (odds + res * k - 1) / (res * k) : 0;          // odds per segment
        const uint64_t sz = (per + SEG_MIN - 1) / SEG_MIN * SEG_MIN;
        seg = (uint32_t)(sz < SEG_MIN ? SEG_MIN : (sz > SEG ? SEG : sz));
    }
    a.seg = seg;
    a.n_seg = odds ? (odds + seg - 1) / seg : 0;
    a.emit_two = lo < 2 && hi >= 2;
    return a;
}

int gen_grid(uint64_t n_seg, int resident) {
    uint64_t g = (uint64_t)(resident > 0 ? resident : 1);
    if (n_seg < g) g = n_seg;
    return (int)(g ? g : 1);
}

}  // namespace

int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

uint64_t l2_bytes() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrL2CacheSize, dev);
        if (n <= 0) n = 1 << 20;
    }
    return (uint64_t)n;
}

cudaError_t launch_gen_small(const DevPlan &pl, uint64_t lo, uint64_t hi, const uint32_t *base,
                             uint32_t n_base, SmallPrime *out, uint64_t cap,
                             unsigned long long *count, cudaStream_t stream) {
    const int res = gen_resident<KIND_SMALL>();
    GenArgs a = make_args(lo, hi, base, n_base, res);
    if (a.n_seg == 0 && !a.emit_two) return cudaSuccess;
    a.kch32 = pl.kch32; a.n_kch32 = pl.n_kch32;
    a.M_start = pl.M_start; a.SL = pl.SL;
    a.o0 = out; a.cap = cap; a.count = count; a.err = pl.stats + ST_ERROR;
    k_gen<KIND_SMALL><<<gen_grid(a.n_seg, res), GEN_THREADS, GEN_SMEM, stream>>>(a);
    return cudaGetLastError();
}

namespace {
// residues of the primes a launch of k_gen<KIND_LIST> over (.., hi] writes: one wave
// of resident CTAs over the count
template <bool P32, bool V>
cudaError_t launch_res_kernel(const GenArgs &a, cudaStream_t stream) {
    static std::atomic<int> res_per_sm{0};
    int per_sm = res_per_sm.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_large_res<P32, V>, RES_THREADS, 0) != cudaSuccess ||
            per_sm <= 0)
            per_sm = 4;
        res_per_sm.store(per_sm, std::memory_order_relaxed);
    }
    k_large_res<P32, V><<<sm_count() * per_sm, RES_THREADS, 0, stream>>>(a);
    return cudaGetLastError();
}
// (a chunk of a plan or a cache lies below 2^32, which is no prime, or above)
cudaError_t launch_res(const GenArgs &a, uint64_t hi, bool with_v, cudaStream_t stream) {
    if (hi > 1ull << 32) return with_v ? launch_res_kernel<false, true>(a, stream) : launch_res_kernel<false, false>(a, stream);
    return with_v ? launch_res_kernel<true, true>(a, stream) : launch_res_kernel<true, false>(a, stream);
}
}  // namespace

cudaError_t launch_gen_large(const DevPlan &pl, bool narrow, uint64_t lo, uint64_t hi,
                             const uint32_t *base, uint32_t n_base, void *p_out, void *r_out,
                             void *v_out, uint64_t cap, unsigned long long *count,
                             cudaStream_t stream) {
    const int res = narrow ? gen_resident<KIND_LARGE32>() : gen_resident<KIND_LIST>();
    GenArgs a = make_args(lo, hi, base, n_base, res);
    if (a.n_seg == 0 && !a.emit_two) return cudaSuccess;
    a.kch32 = pl.kch32; a.n_kch32 = pl.n_kch32;
    a.klimb = pl.klimb; a.n_klimb = pl.n_klimb;
    a.M_start = pl.M_start; a.SL = pl.SL;
    a.o0 = p_out; a.o1 = r_out; a.o2 = v_out;
    a.cap = cap; a.count = count; a.err = pl.stats + ST_ERROR;
    if (narrow) {
        k_gen<KIND_LARGE32><<<gen_grid(a.n_seg, res), GEN_THREADS, GEN_SMEM, stream>>>(a);
        return cudaGetLastError();
    }
    k_gen<KIND_LIST><<<gen_grid(a.n_seg, res), GEN_THREADS, GEN_SMEM, stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_res(a, hi, true, stream);
}

cudaError_t launch_gen_pr(const DevPlan &kp, bool narrow, uint64_t lo, uint64_t hi, const uint32_t *base,
                          uint32_t n_base, void *p_out, void *r_out, uint64_t cap,
                          unsigned long long *count, unsigned long long *err, cudaStream_t stream) {
    const int res = narrow ? gen_resident<KIND_PR32>() : gen_resident<KIND_LIST>();
    GenArgs a = make_args(lo, hi, base, n_base, res);
    if (a.n_seg == 0 && !a.emit_two) return cudaSuccess;
    a.kch32 = kp.kch32; a.n_kch32 = kp.n_kch32;
    a.klimb = kp.klimb; a.n_klimb = kp.n_klimb;
    a.o0 = p_out; a.o1 = r_out;
    a.cap = cap; a.count = count; a.err = err;
    if (narrow) {
        k_gen<KIND_PR32><<<gen_grid(a.n_seg, res), GEN_THREADS, GEN_SMEM, stream>>>(a);
        return cudaGetLastError();
    }
    k_gen<KIND_LIST><<<gen_grid(a.n_seg, res), GEN_THREADS, GEN_SMEM, stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_res(a, hi, false, stream);
}

cudaError_t launch_gen_list(uint64_t lo, uint64_t hi, const uint32_t *base, uint32_t n_base,
                            uint64_t *out, uint64_t cap, unsigned long long *count,
                            unsigned long long *err, cudaStream_t stream) {
    const int res = gen_resident<KIND_LIST>();
    GenArgs a = make_args(lo, hi, base, n_base, res);
    if (a.n_seg == 0 && !a.emit_two) return cudaSuccess;
    a.o0 = out; a.cap = cap; a.count = count; a.err = err;
    k_gen<KIND_LIST><<<gen_grid(a.n_seg, res), GEN_THREADS, GEN_SMEM, stream>>>(a);
    return cudaGetLastError();
}

namespace {
__global__ void k_kmodp(const uint64_t *p, uint64_t n, uint64_t *r, const uint32_t *kch32,
                        uint32_t n32, const uint32_t *klimb, uint32_t n_limb) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t q = p[i];
        if (q < (1ull << 31)) {
            uint32_t q32 = (uint32_t)q;
            uint32_t pinv = mont32_neg_inv(q32);
            r[i] = kmodp32(q32, pinv, mont32_r1(q32), mont32_r2(q32), kch32, n32);
        } else if (q >> 32) {
            r[i] = res_k_mod_p<false>(res_mod<false>(q), klimb, n_limb);
        } else {
            r[i] = res_k_mod_p<true>(res_mod<true>(q), klimb, n_limb);
        }
    }
}
}  // namespace

cudaError_t launch_kmodp(const DevPlan &pl, const uint64_t *p, uint64_t n, uint64_t *r,
                         cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    k_kmodp<<<(unsigned)blocks, 256, 0, stream>>>(p, n, r, pl.kch32, pl.n_kch32, pl.klimb,
                                                   pl.n_klimb);
    return cudaGetLastError();
}

}  // namespace cs
