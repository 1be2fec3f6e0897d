// bn_fx.cuh -- fixed-point arithmetic in integers: rounding of the exact 128-bit sums (64
// fraction bits, two's complement), and powers of ten.  Compiles as plain C++ too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define BN_FX_FN __host__ __device__ __forceinline__
#else
#define BN_FX_FN inline
#endif
#ifdef __CUDA_ARCH__
#define BN_CLZ(x) __clzll((long long)(x))
#define BN_MULHI(a, b) __umul64hi(a, b)
#else
#define BN_CLZ(x) ((x) ? __builtin_clzll(x) : 64)
#define BN_MULHI(a, b) (uint64_t)(((unsigned __int128)(a) * (b)) >> 64)
#endif

namespace bn {

// The bits of u / ln 10 as an FP64 -- the low word rounded to 53 bits, the sum hi + lo 2^-64
// rounded, the quotient rounded, all to nearest even -- in integers: the two conversions,
// the addition and the division are eight operations of an FP64 pipe that takes 1.7 us for one
// operation of a million entries (a build of 29.4 M entries: 0.51 ms for k_assemble, 0.34
// in integers).  |u| < 2^115.  The quotient is a multiplication by Z, the reciprocal of ln 10's
// mantissa, a remainder and one correction (Granlund and Montgomery, division by invariant
// integers); a quotient of two 53-bit numbers never lies half way.
BN_FX_FN uint64_t fx_div_ln10(unsigned __int128 u)
{
    constexpr uint64_t L = 0x126bb1bbb55516ull;                 // the FP64 nearest ln 10 is L 2^-51
    constexpr uint64_t Z = (uint64_t)(((unsigned __int128)1 << 116) / L);
    uint64_t hi = (uint64_t)(u >> 64), lo = (uint64_t)u;
    if (lo >> 53) {
        const int s = 11 - BN_CLZ(lo);                          // bits that go
        const uint64_t t = lo + ((1ull << (s - 1)) - 1 + ((lo >> s) & 1u));
        hi += t < lo;
        lo = t & ~((1ull << s) - 1);
    }
    const uint64_t sign = hi & 0x8000000000000000ull;
    if (sign) {
        lo = 0 - lo;
        hi = ~hi + (lo == 0);
    }
    if (!(hi | lo)) return 0;
    // 64 leading bits, and those below
    const int zh = BN_CLZ(hi), z = hi ? zh : 64 + BN_CLZ(lo);
    const uint64_t top = z >= 64 ? lo << (z - 64) : z ? (hi << z) | (lo >> (64 - z)) : hi;
    const uint64_t rest = z >= 64 ? 0 : lo << z;
    const uint32_t low = (uint32_t)top & 0x7ffu;
    uint64_t M = top >> 11;
    int e = 1074 + 10 - z;                                      // exponent field, less one, + 51 - 53
    M += low > 0x400u || (low == 0x400u && (rest || (M & 1u)));
    if (M >> 53) {
        M >>= 1;
        ++e;
    }
    const int s = M >= L ? 52 : 53;
    uint64_t q = BN_MULHI(M << 11, Z) >> (63 - s);
    const uint64_t r = (M << s) - q * L;                        // below 2 L
    q += (2 * r > L) + (2 * r > 3 * L);
    return (((uint64_t)(e - s + 52) << 52) + q) | sign;         // (a carry of q goes to the exponent)
}

// 2^(-j / 64), 2^(-j / 4096) and 2^(-j / 262144), j < 64, with 63 fractional bits, from the
// exponential series in integer arithmetic
struct Exp2Tables {
    uint64_t v[3][64];
};
constexpr uint64_t LN2_64 = 0xB17217F7D1CF79ACull;        // ln 2 in 2^-64
constexpr uint64_t mulhi_c(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
constexpr Exp2Tables make_exp2()
{
    Exp2Tables T{};
    for (int t = 0; t < 3; ++t)
        for (int j = 0; j < 64; ++j) {
            // e^-z, z = ln 2 * j / 64^(t + 1), as sum (-z)^k / k! in 2^-64 with 128-bit sums
            const uint64_t x = (uint64_t)j << (58 - 6 * t);                  // j / 64^(t + 1) in 2^-64
            const uint64_t z = mulhi_c(x, LN2_64);
            unsigned __int128 pos = (unsigned __int128)1 << 64, neg = 0;
            uint64_t term = z;
            for (int k = 1; k < 24; ++k) {
                if (k & 1) neg += term;
                else pos += term;
                term = mulhi_c(term, z) / (uint64_t)(k + 1);
            }
            T.v[t][j] = (uint64_t)((pos - neg + 1) >> 1);
        }
    return T;
}
// 10^-d in 2^-59 for d in [0, 1] given in 2^-60, within 2^-55 of itself (cut off at 2^-58 it is
// 2^-54.7) and below 1, so that 32 of them fit 64 bits: d log2 10 = whole + three table digits
// of six bits + a rest below 2^-18, whose 2^-r = 1 - z + z^2 / 2 up to z^3 / 6 < 2^-58
BN_FX_FN uint64_t exp10_fx(uint64_t d, const uint64_t (&T)[3][64])
{
    constexpr uint64_t LOG2_10 = 0x6A4D3C25E68DC57Full;                      // log2 10 in 2^-61
    const uint64_t y = BN_MULHI(d, LOG2_10);                                 // in 2^-57
    const uint32_t whole = (uint32_t)(y >> 57);
    const uint64_t t1 = T[0][(y >> 51) & 63], t2 = T[1][(y >> 45) & 63], t3 = T[2][(y >> 39) & 63];
    const uint64_t r = y & ((1ull << 39) - 1);                               // in 2^-57, below 2^-18
    const uint64_t z = BN_MULHI(r << 25, LN2_64);                            // in 2^-82, below 2^63.5
    const uint32_t zh = (uint32_t)(z >> 32);                                 // z in 2^-50
    const uint64_t sq = (uint64_t)zh * zh;                                   // z^2 in 2^-100
    // 1 - z + z^2 / 2 in 2^-63, less one unit
    const uint64_t e = ((1ull << 63) - 1) - (z >> 19) + (sq >> 38);
    uint64_t p = BN_MULHI(t1, t2) << 1;                                      // 2^-63 each
    p = BN_MULHI(p, t3) << 1;
    p = BN_MULHI(p, e);                                                      // 2^-62
    return (p >> 3) >> whole;                                                // 2^-59
}

}  // namespace bn
#undef BN_CLZ
#undef BN_MULHI
