// soft64.h -- binary64 multiply and add on the integer pipes, each the same
// bits as the IEEE operation (round to nearest even) wherever it reports that
// it applies.  For kernels bound by the binary64 unit, which on GB300 holds a
// warp instruction 64 cycles per sub-partition: these take the integer and
// binary32 pipes instead and run beside it.
//
// Also compiles as plain C++ (the tests compare it with the host's arithmetic).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define AEB_HD __host__ __device__ __forceinline__
#else
#include <string.h>
#define AEB_HD inline
#endif

namespace aeb {

AEB_HD uint64_t bits_of(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    __builtin_memcpy(&b, &x, 8);
    return b;
#endif
}
AEB_HD double of_bits(uint32_t hi, uint32_t lo)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = ((uint64_t)hi << 32) | lo;
    double x;
    __builtin_memcpy(&x, &b, 8);
    return x;
#endif
}

// A factor in the form the multiply takes: its 53-bit significand at the top
// of 64 bits, and what its sign and exponent add to the product's high word.
// The factor is normal with an exponent in [-256, 256] (`soft_factor_ok`).
struct SoftFactor {
    uint32_t lo, hi, ex;
};
AEB_HD bool soft_factor_ok(double m)
{
    const uint32_t e = ((uint32_t)(bits_of(m) >> 32) >> 20) & 0x7ffu;
    return e >= 1023 - 256 && e <= 1023 + 256;
}
AEB_HD SoftFactor soft_factor(double m)
{
    const uint64_t b = bits_of(m);
    const uint64_t s = (b << 11) | (uint64_t(1) << 63);
    SoftFactor f;
    f.lo = (uint32_t)s;
    f.hi = (uint32_t)(s >> 32);
    f.ex = ((uint32_t)(b >> 32) & 0xfff00000u) - (1023u << 20);
    return f;
}

// a m.  The result is the product where a is normal with an exponent in
// [-255, 256] (the product then is normal too); otherwise it is not, and
// soft_bad(range) holds (`range` accumulates over operations, start at 0).
AEB_HD bool soft_bad(uint32_t range) { return (range >> 30) != 0; }
AEB_HD double soft_mul(double a, const SoftFactor &m, uint32_t &range)
{
    const uint64_t b = bits_of(a);
    const uint32_t ah = (uint32_t)(b >> 32), al = (uint32_t)b;
    // exponent field in [0x300, 0x500): twice the high word, less the sign
    range |= ah + ah - 0x60000000u;
    // 53 x 64 bits: H = the top 64 of P = significand(a) * (m.hi:m.lo), in
    // [2^51, 2^53); l = the rest
    const uint32_t mh = (ah & 0xfffffu) | 0x100000u;
    const uint64_t p0 = (uint64_t)al * m.lo;
    const uint64_t p1 = (uint64_t)al * m.hi + (p0 >> 32);
    const uint64_t p2 = (uint64_t)mh * m.lo + (uint32_t)p1;
    uint64_t h = (uint64_t)mh * m.hi + (p1 >> 32) + (p2 >> 32);
    uint64_t l = (p2 << 32) | (uint32_t)p0;
    uint32_t ex = (ah & 0xfff00000u) + m.ex;
    if (!(h >> 52)) {  // a product of significands below 2
        h = (h << 1) | (l >> 63);
        l <<= 1;
        ex -= 1u << 20;
    }
    // up if l > 2^63, or l == 2^63 and h is odd: the carry out of the sum
    const uint64_t c = l + (0x7fffffffffffffffull + (h & 1));
    h += c < l ? 1u : 0u;
    return of_bits((uint32_t)(h >> 32) + ex, (uint32_t)h);
}

// a + b where a's exponent (in [-1000, 1000]) exceeds b's by 0 to 31 (WIDE: to 63), both are
// normal and the sum is in a's binade or the next on either side; otherwise the
// result is not the sum and soft_bad(range) holds.
template <bool WIDE>
AEB_HD double soft_add(double a, double b, uint32_t &range)
{
    const uint64_t x = bits_of(a), y = bits_of(b);
    const uint32_t xh = (uint32_t)(x >> 32), yh = (uint32_t)(y >> 32);
    const uint32_t d = ((xh >> 20) & 0x7ffu) - ((yh >> 20) & 0x7ffu), d5 = d & 31u;
    // b's significand, negated if the signs differ, shifted to a's scale
    const uint32_t neg = (uint32_t)((int32_t)(xh ^ yh) >> 31);
    uint64_t m = ((uint64_t)((yh & 0xfffffu) | 0x100000u) << 32) | (uint32_t)y;
    m = (m ^ (((uint64_t)neg << 32) | neg)) + (neg & 1u);
    const uint32_t ml = (uint32_t)m;
    const int32_t mh = (int32_t)(uint32_t)(m >> 32);
#ifdef __CUDA_ARCH__
    uint32_t qlo = __funnelshift_r(ml, (uint32_t)mh, d5);
    uint32_t f = __funnelshift_lc(0u, ml, 32u - d5);  // the 32 bits below a's last
#else
    uint32_t qlo = (uint32_t)(m >> d5);
    uint32_t f = d5 ? ml << (32u - d5) : 0u;
#endif
    uint32_t qhi = (uint32_t)(mh >> d5);
    uint32_t rest = 0;  // whether bits below f are set
    if (WIDE && (d & 32u)) {
        rest = f != 0u ? 1u : 0u;
        f = qlo;
        qlo = qhi;
        qhi = neg;
    }
    // on the packed form: the significand's carry or borrow moves the exponent
    uint64_t s = x + (((uint64_t)qhi << 32) | qlo);
    bool ok = d < (WIDE ? 64u : 32u) && (yh & 0x7ff00000u) != 0u;
    const uint32_t step = (uint32_t)(s >> 32) - (xh & 0xfff00000u);
    if (step >> 20) {  // another binade (~30 times a rollout)
        constexpr uint64_t kField = 0xfffffffffffffull;
        const uint64_t field = s & kField;
        if (step >> 20 == 1u) {  // next: one bit more to round off
            rest |= f & 1u;
            f = (f >> 1) | ((uint32_t)s << 31);
            s = (s & ~kField) | (field >> 1);
        } else {  // previous: one bit more of the sum
            ok = ok && step >> 20 == 0xfffu && (field >> 51);
            s = (s & ~kField) | (((field << 1) | (f >> 31)) & kField);
            f <<= 1;
        }
    }
    // up if the fraction is above a half, or a half and s is odd
    s += f > 0x80000000u - (((uint32_t)s & 1u) | rest) ? 1u : 0u;
    range |= ok ? 0u : 0x80000000u;
    return of_bits((uint32_t)(s >> 32), (uint32_t)s);
}

}  // namespace aeb
