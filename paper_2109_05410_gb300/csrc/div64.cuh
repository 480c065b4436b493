// div64.cuh -- FP64 values from FP32 operands without the FP64 pipe, which
// issues one warp instruction every 16 clocks per SM on GB300: widening a
// float, and dividing a double by a float with IEEE rounding, both in
// integer and FP32 instructions.  Host code compiles it too.
#pragma once
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define OOC_HD __host__ __device__ __forceinline__
#else
#define OOC_HD inline
#endif

namespace ooc {

template <typename To, typename From>
OOC_HD To bits_as(From v)
{
    static_assert(sizeof(To) == sizeof(From), "bits_as");
    To t;
    memcpy(&t, &v, sizeof(t));
    return t;
}

// (double) v: zeros and normal values by moving the bits, the others by the
// conversion.
OOC_HD double widen(float v)
{
    const uint32_t b = bits_as<uint32_t>(v), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u) {
        const uint64_t hi = (b & 0x80000000u) | ((m >> 3) + 0x38000000u);
        return bits_as<double>(hi << 32 | (uint64_t)(b << 29));
    }
    if (m == 0u)
        return bits_as<double>((uint64_t)b << 32);
    return (double)v;
}

// The 24-bit significand of a normal k as a float in [1, 2).
OOC_HD float significand(float k) { return bits_as<float>((bits_as<uint32_t>(k) & 0x007fffffu) | 0x3f800000u); }

// g / (double) k, correctly rounded (nearest, ties to even), given
// rcp = 1 / significand(k) to within 2^-22: schoolbook long division of the
// 53-bit significand by the 24-bit one, digit by digit (30 bits in two
// estimates, then 23 bits), each estimate corrected by its exact remainder.
// Zero numerators give a signed zero; denormal, infinite and NaN operands and
// quotients near the exponent range's ends take the division itself.
OOC_HD double div_f64_f32(double g, float k, float rcp)
{
    const uint64_t gb = bits_as<uint64_t>(g);
    const uint32_t kb = bits_as<uint32_t>(k);
    const uint32_t ge = (uint32_t)(gb >> 52) & 0x7ffu, ke = (kb >> 23) & 0xffu;
    const uint64_t sign = (gb ^ (uint64_t)kb << 32) & 0x8000000000000000ull;
    const bool kn = ke - 1u < 254u;
    if (kn && gb << 1 == 0)
        return bits_as<double>(sign);
    // quotient exponent (biased): ge - ke + 127, one less if g's significand
    // is the smaller
    if (!kn || ge - 256u >= 1536u)
        return g / (double)k;
    uint64_t m = (gb & 0x000fffffffffffffull) | 0x0010000000000000ull;
    const uint32_t d = (kb & 0x007fffffu) | 0x00800000u;
    uint32_t e = ge + 127u - ke;
    if (m < (uint64_t)d << 29) {
        m <<= 1;
        --e;
    }
    // q1 = floor(m / d), in [2^29, 2^30).  First estimate in steps of 2^7:
    // m / 2^30 (24 bits) times rcp is m / (2^7 d), rounded by adding 2^23.
    const float magic = 8388608.0f, magic2 = 12582912.0f;
    const uint32_t a = bits_as<uint32_t>((float)(uint32_t)(m >> 30) * rcp + magic) - 0x4b000000u;
    uint32_t q1 = a << 7;
    const int64_t r1 = (int64_t)(m - (uint64_t)q1 * d);  // |r1| < 2^10 d
    const float f1 = (float)(int32_t)(r1 >> 4) * (rcp * 1.9073486328125e-6f);  // r1 / d, rcp 2^4 / 2^23
    const int32_t b = (int32_t)bits_as<uint32_t>(f1 + magic2) - 0x4b400000;
    q1 += (uint32_t)b;
    int32_t r = (int32_t)((uint32_t)r1 - (uint32_t)b * d);  // in (-2 d, 2 d)
    if (r < 0) {
        r += (int32_t)d;
        --q1;
    }
    if (r >= (int32_t)d) {
        r -= (int32_t)d;
        ++q1;
    }
    // q2 = floor(r 2^23 / d), in [0, 2^23)
    uint32_t q2 = bits_as<uint32_t>((float)r * rcp + magic) - 0x4b000000u;
    int32_t t = (int32_t)(((uint32_t)r << 23) - q2 * d);  // in (-4 d, 4 d)
    if (t < -(int32_t)d) {
        t += 2 * (int32_t)d;
        q2 -= 2u;
    }
    if (t < 0) {
        t += (int32_t)d;
        --q2;
    }
    if (t >= 2 * (int32_t)d) {
        t -= 2 * (int32_t)d;
        q2 += 2u;
    }
    if (t >= (int32_t)d) {
        t -= (int32_t)d;
        ++q2;
    }
    uint64_t q = ((uint64_t)q1 << 23) + q2;
    if (2 * t > (int32_t)d || (2 * t == (int32_t)d && (q2 & 1u)))
        ++q;  // 2^53 carries into the exponent
    return bits_as<double>(sign | (((uint64_t)(e - 1u) << 52) + q));
}

}  // namespace ooc
