// Jump-ahead of the 32-bit generators by a fixed number of draws, the words that
// so many single draws leave, bit for bit.
//
// Tausworthe words.  With k = 31, 29, 28, q = S1 and s = S3, a word is 32
// consecutive bits b_n, b_{n+1}, ... (b_n the highest) of the sequence
// b_{m+k} = b_m ^ b_{m+q}, and a step moves it s bits on (a seed's 32 - k lowest
// bits are not part of the sequence, and no step reads them).  D steps move it
// m = s D bits on, and b_{n+m} is the sum of the b_{n+i} whose x^i occurs in
// x^m mod x^k + x^q + 1.  So the jumped word is the xor of the windows at those
// i < k, all inside the 64 bits that follow b_n: two applications of the
// recurrence form these, and about 15 funnel shifts and their xors the word.
// The polynomials are compile-time constants.  A jump of the three words is about
// 110 instructions in registers.  (Products with 4-bit groups from tables in
// shared memory are 84 instructions, 24 of them conflicting loads, and the tables
// cost small systems' blocks their room: ld_run of 1e4 Hybrid Taus oscillators
// 76.0 -> 72.0 us for 1000 steps, 16.5 -> 14.6 for 50.)
//
// LCG word: one multiply and one add.
#pragma once

#include "device.cuh"

namespace gb {

// x^m mod x^k + x^q + 1 over GF(2); bit i is the coefficient of x^i.
__host__ __device__ constexpr uint32_t gf2_mulmod(uint32_t u, uint32_t v, int k, int q)
{
    uint64_t p = 0;   // degree at most 2k - 2 <= 60
    for (; v; v &= v - 1) {
        const uint32_t low = v & (0u - v);
        p ^= (uint64_t)u * low;   // u x^i
    }
    // x^{k+i} = x^{q+i} + x^i, twice: the first leaves a degree of at most k - 2 + q
    const uint64_t mask = (1ull << k) - 1;
    for (int r = 0; r < 2; ++r) {
        const uint64_t h = p >> k;
        p = (p & mask) ^ h ^ (h << q);
    }
    return (uint32_t)p;
}

__host__ __device__ constexpr uint32_t gf2_xpow(uint64_t m, int k, int q)
{
    uint32_t r = 1, b = 2;
    for (; m; m >>= 1) {
        if (m & 1) r = gf2_mulmod(r, b, k, q);
        b = gf2_mulmod(b, b, k, q);
    }
    return r;
}

// One word, moved on by the number of bits of the polynomial (a constant after
// inlining, or not).
template <int K, int Q>
__device__ __forceinline__ uint32_t taus_word_jump(uint32_t y, uint32_t poly)
{
    // bits b_n .. b_{n+63} from the K highest of y: the first application is
    // right up to bit 2K - Q - 1, which the second reads no further than
    const uint64_t z = (uint64_t)(y & (0xFFFFFFFFu << (32 - K))) << 32;
    const uint64_t w = z | ((z ^ (z << Q)) >> K);
    static_assert(63 - K + Q <= 2 * K - Q - 1, "two applications give 64 bits");
    const uint64_t u = z | ((w ^ (w << Q)) >> K);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) r ^= __funnelshift_l(lo, hi, i) & (0u - ((poly >> i) & 1u));
    return r;
}

struct LcgJump {
    uint32_t a, c;   // x -> a x + c
};

__host__ __device__ constexpr LcgJump lcg_jump(uint64_t d)
{
    LcgJump r{1u, 0u}, m{1664525u, 1013904223u};
    for (; d; d >>= 1) {
        if (d & 1) r = LcgJump{m.a * r.a, m.a * r.c + m.c};
        m = LcgJump{m.a * m.a, m.a * m.c + m.c};
    }
    return r;
}

template <uint64_t D>
__device__ __forceinline__ void jump_ahead(uint32_t& x)
{
    constexpr LcgJump l = lcg_jump(D);
    x = l.a * x + l.c;
}

template <uint64_t D>
__device__ __forceinline__ void jump_ahead(uint4& y)
{
    constexpr uint32_t p1 = gf2_xpow(12 * D, 31, 13), p2 = gf2_xpow(4 * D, 29, 2), p3 = gf2_xpow(17 * D, 28, 3);
    y.x = taus_word_jump<31, 13>(y.x, p1);
    y.y = taus_word_jump<29, 2>(y.y, p2);
    y.z = taus_word_jump<28, 3>(y.z, p3);
    jump_ahead<D>(y.w);
}

// A jump whose distance is known at run time.
struct Jump {
    uint32_t p[3];   // the Tausworthe words' polynomials
    LcgJump l;
};

inline Jump jump_of(uint64_t d)
{
    return Jump{{gf2_xpow(12 * d, 31, 13), gf2_xpow(4 * d, 29, 2), gf2_xpow(17 * d, 28, 3)}, lcg_jump(d)};
}

// The jump by both distances.
inline Jump jump_sum(const Jump& a, const Jump& b)
{
    return Jump{{gf2_mulmod(a.p[0], b.p[0], 31, 13), gf2_mulmod(a.p[1], b.p[1], 29, 2),
                 gf2_mulmod(a.p[2], b.p[2], 28, 3)},
                LcgJump{a.l.a * b.l.a, a.l.a * b.l.c + a.l.c}};
}

__device__ __forceinline__ void jump_ahead(uint32_t& x, const Jump& j) { x = j.l.a * x + j.l.c; }
__device__ __forceinline__ void jump_ahead(uint4& y, const Jump& j)
{
    y.x = taus_word_jump<31, 13>(y.x, j.p[0]);
    y.y = taus_word_jump<29, 2>(y.y, j.p[1]);
    y.z = taus_word_jump<28, 3>(y.z, j.p[2]);
    jump_ahead(y.w, j);
}

}  // namespace gb
