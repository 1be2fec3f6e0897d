// bn_fx.cuh -- rounding of the exact 128-bit fixed-point sums (64 fraction bits, two's
// complement), in integers.  Compiles as plain C++ too.
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

}  // namespace bn
#undef BN_CLZ
#undef BN_MULHI
