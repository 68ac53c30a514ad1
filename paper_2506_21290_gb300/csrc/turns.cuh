// Phases in turns and their cosines, in integer arithmetic.
//
// The correlations and S(q) are means of cos(q . d) over fixed-point
// displacements d = n h (n integer, h = L / 2^32).  In FP64 such a cosine takes
// some 33 operations of a pipe that does 2 per SM and cycle on this part; the
// integer units do 64 multiplies per cycle.  So:
//
//   phase:  q . d / 2 pi turns = sum over axes of kappa n with
//           kappa = q h / 2 pi.  Whole turns do not matter, so kappa is kept as
//           the 96 bits of its fraction and the sum is taken modulo one turn in
//           64 bits.  kappa is exact to 2^-96 for any finite q (its FP64 value,
//           times h, times 1 / 2 pi to 2304 bits), so the phase is exact to
//           2^-62 turns; an FP64 phase carries its own size times 2^-53.
//   cosine: the Taylor series of cos over a quarter turn in t = (4 x)^2, twelve
//           terms (the next one is 2^-63), 64-bit fixed point, the terms
//           below 2^-25 in 32 bits.  Largest error 2^-57.8 (20000 phases
//           against 200-bit arithmetic), then rounded to 2^-53: an FP64 cosine
//           is as far off (half a unit of 2^-53).
//
// Sums of these integers are exact, whatever their order.  Against extended
// precision (64 to 2000 molecules, wavevectors near 7.4 and 5.1): F_s and
// F_s^cm per particle within 4e-17 to 7e-17 of their norm (FP64 cosines: 1.4e-16
// to 2.2e-16), S(q) 2e-16 to 2.5e-16 (FP64: 1e-15 to 4e-15).
#pragma once

#include <cstdint>

#include "energy.h"

namespace flipmc {

// 1 / (2 pi) and 1 / (6 pi) as binary fractions, 32 bits per word, first word first
__constant__ const uint32_t kInv2Pi[72] = {
    0x28BE60DBu, 0x9391054Au, 0x7F09D5F4u, 0x7D4D3770u, 0x36D8A566u, 0x4F10E410u, 0x7F9458EAu, 0xF7AEF158u,
    0x6DC91B8Eu, 0x909374B8u, 0x01924BBAu, 0x82746487u, 0x3F877AC7u, 0x2C4A69CFu, 0xBA208D7Du, 0x4BAED121u,
    0x3A671C09u, 0xAD17DF90u, 0x4E64758Eu, 0x60D4CE7Du, 0x272117E2u, 0xEF7E4A0Eu, 0xC7FE25FFu, 0xF7816603u,
    0xFBCBC462u, 0xD6829B47u, 0xDB4D9FB3u, 0xC9F2C26Du, 0xD3D18FD9u, 0xA797FA8Bu, 0x5D49EEB1u, 0xFAF97C5Eu,
    0xCF41CE7Du, 0xE294A4BAu, 0x9AFED7ECu, 0x47E35742u, 0x1580CC11u, 0xBF1EDAEAu, 0xFC33EF08u, 0x26BD0D87u,
    0x6A78E458u, 0x57B986C2u, 0x19666157u, 0xC5281A10u, 0x237FF620u, 0x135CC9CCu, 0x41818555u, 0xB29CEA32u,
    0x58389EF0u, 0x231AD1F1u, 0x0670D9F3u, 0x773A024Au, 0xA0D6711Du, 0xA2E58729u, 0xB76BD134u, 0x55C6414Fu,
    0xA97FC1C1u, 0x4FDF8CFAu, 0x0CB0B793u, 0xE60C9F6Eu, 0xF0CF49BBu, 0xDAC797BEu, 0x27CE87CDu, 0x72BC9FC7u,
    0x61FC4864u, 0x1F1F091Au, 0xBE9BB55Du, 0xCB4C10CEu, 0xC571852Du, 0x674670F0u, 0xB12B5053u, 0x4B174003u};
__constant__ const uint32_t kInv6Pi[72] = {
    0x0D94CAF3u, 0xDBDB01C3u, 0x7FADF1FCu, 0x29C467D0u, 0x12483722u, 0x1A5AF6B0u, 0x2A86C84Eu, 0x528FA5C8u,
    0x24985E84u, 0xDADBD192u, 0xAB30C3E8u, 0xD626CC2Du, 0x152D28EDu, 0x0EC3789Au, 0x93602F29u, 0xC3E4F060u,
    0x68CD0958u, 0x8F07F530u, 0x1A217C84u, 0xCAF19A29u, 0xB7B5B2A0u, 0xFA7F6E04u, 0xED54B755u, 0x52807756u,
    0xA943EC20u, 0xF22B8917u, 0xF3C48A91u, 0x4350EB79u, 0xF145DA9Du, 0xE287FE2Eu, 0x746DFA3Bu, 0x53A87ECAu,
    0x4515EF7Fu, 0x4B86E193u, 0x88FF9D4Eu, 0xC2A11D16u, 0x072AEEB0u, 0x950A48F8u, 0xFEBBFA58u, 0x0CE9AF2Du,
    0x237DA172u, 0xC7E88240u, 0xB3222072u, 0x970D5E05u, 0x612AA760u, 0x06744344u, 0x15D5D71Cu, 0x90DEF8BBu,
    0x72BD8A50u, 0x0BB39B50u, 0x577AF351u, 0x27BE00C3u, 0x8AF225B4u, 0x8BA1D7B8u, 0x927945BCu, 0x1C976B1Au,
    0x8DD54095u, 0xC54A8453u, 0x59903D31u, 0x4CAEDFCFu, 0xA59A6DE9u, 0x48ED3294u, 0xB7EF8299u, 0xD0E98A97u,
    0xCB541821u, 0x5FB50308u, 0xEA33E71Fu, 0x43C4059Au, 0x41D081B9u, 0xCD177AFAu, 0xE5B91AC6u, 0x6E5D1556u};

// The 96-bit fraction of q h c with c the fraction held in `inv`, |q| and h FP64.
__device__ inline void turn_fraction(double q, double h, const uint32_t *inv, uint32_t out[3])
{
    out[0] = out[1] = out[2] = 0;
    // q and h as 53-bit integers times powers of two (subnormals included)
    auto split = [](double x, uint64_t &m, int &e) {
        const uint64_t b = (uint64_t)__double_as_longlong(x);
        const int ex = (int)((b >> 52) & 0x7FF);
        m = (b & 0xFFFFFFFFFFFFFull) | (ex ? 1ull << 52 : 0ull);
        e = (ex ? ex : 1) - 1075;
    };
    uint64_t mq, mh;
    int eq, eh;
    split(fabs(q), mq, eq);
    split(h, mh, eh);
    if (mq == 0) return;
    const uint64_t p0 = mq * mh, p1 = __umul64hi(mq, mh);
    const uint32_t p[4] = {(uint32_t)p0, (uint32_t)(p0 >> 32), (uint32_t)p1, (uint32_t)(p1 >> 32)};
    const int E = eq + eh;                   // q h = p 2^E
    // word j of c times p 2^E is a whole number while 32 (j + 1) <= E; nine
    // words from there leave less than 2^-96 behind
    const int j0 = E > 0 ? min(E >> 5, 63) : 0;
    uint32_t w[14] = {};                     // p times the nine words, lowest word first
    for (int j = 0; j < 9; ++j) {
        const uint64_t c = inv[j0 + 8 - j];
        uint64_t carry = 0;
        for (int k = 0; k < 4; ++k) {
            const uint64_t v = c * p[k] + w[j + k] + carry;
            w[j + k] = (uint32_t)v;
            carry = v >> 32;
        }
        w[j + 4] = (uint32_t)carry;
    }
    // q h c = w 2^(E - 32 (j0 + 9)) modulo 1: its bits -1 .. -96
    const int s = 32 * (j0 + 9) - E - 96;
    for (int k = 0; k < 3; ++k) {
        const int at = s + 32 * k, word = at >> 5, sh = at & 31;
        if (at < 0 || word > 13) continue;
        const uint64_t hi = word + 1 <= 13 ? w[word + 1] : 0u;
        out[k] = (uint32_t)((hi << 32 | w[word]) >> sh);
    }
    if (q < 0.0) {
        const uint64_t lo = 0ull - ((uint64_t)out[1] << 32 | out[0]);
        out[2] = 0u - out[2] - ((out[0] | out[1]) != 0u);
        out[0] = (uint32_t)lo;
        out[1] = (uint32_t)(lo >> 32);
    }
}

__device__ inline Turns make_turns(const double *q, double h, const uint32_t *inv)
{
    Turns t;
    t.bias = 0;
    t.bad = 0;
    for (int ax = 0; ax < 3; ++ax) {
        uint32_t f[3] = {0, 0, 0};
        if (isfinite(q[ax])) turn_fraction(q[ax], h, inv, f);
        else t.bad = 1;
        t.k0[ax] = f[0];
        t.k1[ax] = f[1];
        t.k2[ax] = f[2];
        // 2^31 quanta: the 96 bits shifted left by 31, the highest 64 kept
        t.bias += (((uint64_t)f[1] << 32 | f[0]) >> 1) | (uint64_t)(f[2] & 1u) << 63;
    }
    return t;
}

// phase of the displacement (x, y, z) quanta, unsigned, in units of 2^-64 turns
__device__ __forceinline__ uint64_t turn_phase(const Turns &t, uint32_t x, uint32_t y, uint32_t z)
{
    uint64_t p = (uint64_t)x * t.k1[0];
    p += (uint64_t)y * t.k1[1];
    p += (uint64_t)z * t.k1[2];
    p += (uint64_t)__umulhi(x, t.k0[0]);
    p += (uint64_t)__umulhi(y, t.k0[1]);
    p += (uint64_t)__umulhi(z, t.k0[2]);
    return p + ((uint64_t)(x * t.k2[0] + y * t.k2[1] + z * t.k2[2]) << 32);
}

// the same of multiples of 2^32 quanta (displacements beyond half a box)
__device__ __forceinline__ uint64_t turn_phase_boxes(const Turns &t, int x, int y, int z)
{
    auto one = [](int n, uint32_t k1, uint32_t k0) { return (uint64_t)(int64_t)n * ((uint64_t)k1 << 32 | k0); };
    return one(x, t.k1[0], t.k0[0]) + one(y, t.k1[1], t.k0[1]) + one(z, t.k1[2], t.k0[2]);
}

// the highest 64 bits of x z, at most 2 too small
__device__ __forceinline__ uint64_t mul_hi(uint64_t x, uint64_t z)
{
    const uint32_t xh = (uint32_t)(x >> 32), xl = (uint32_t)x, zh = (uint32_t)(z >> 32), zl = (uint32_t)z;
    return (uint64_t)xh * zh + __umulhi(xh, zl) + __umulhi(xl, zh);
}

// cos(2 pi p / 2^64) in units of 2^-53 (cos 0 is exactly 2^53).
__device__ __forceinline__ long long cos_turn(uint64_t p)
{
    // fold to a quarter turn: cos is even, and cos(1/2 - x) = -cos x
    uint64_t a = (long long)p < 0 ? 0ull - p : p;
    const bool neg = a > 1ull << 62;
    if (neg) a = (1ull << 63) - a;
    // 4 x, 64 fraction bits (the quarter turn itself one unit short)
    const uint64_t y = (a - (a >> 62)) << 2;
    const uint32_t yh = (uint32_t)(y >> 32), yl = (uint32_t)y;
    const uint64_t t = (uint64_t)yh * yh + 2ull * __umulhi(yh, yl);
    const uint32_t th = (uint32_t)(t >> 32);
    // (pi/2)^(2k) / (2k)!: k = 11 .. 7 with 59 fraction bits, k = 6 .. 1 with 63
    uint32_t s = 11u;
    s = 1982u - __umulhi(th, s);
    s = 305201u - __umulhi(th, s);
    s = 37850200u - __umulhi(th, s);
    s = 3681626018u - __umulhi(th, s);
    uint64_t r = 4345015070408ull - ((uint64_t)th * s >> 28);
    r = 232447812895316ull - mul_hi(t, r);
    r = 8478679513545403ull - mul_hi(t, r);
    r = 192431645064167232ull - mul_hi(t, r);
    r = 2339688245777237863ull - mul_hi(t, r);
    r = 11378879155978302162ull - mul_hi(t, r);
    r = (1ull << 63) - mul_hi(t, r);
    const long long v = (long long)((r + 512) >> 10);
    return neg ? -v : v;
}

}  // namespace flipmc
