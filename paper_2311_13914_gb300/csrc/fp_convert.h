// fp_convert.h -- float <-> double by integer arithmetic, bit for bit what the
// conversions give (round to nearest even, NaN quieted).  GB300 issues a
// conversion through the FP64 pipe, where it takes 64 clocks a warp and scheduler
// like a DFMA; the shifts and adds below take about ten.  A conversion left in
// for the rare cases would be predicated off and still take its slot, so those are
// done with integers too.  The passes over FP32 V-cycle vectors in the FP64 PCG
// spent a third of their FP64 slots on conversions (256x256x64 nodes: 99 -> 69 us
// for the z statistics, 57 -> 41 for the direction, 104 -> 88 for x and r).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define BD_FP_FN __host__ __device__ __forceinline__
#else
#define BD_FP_FN inline
#endif

namespace bd {

BD_FP_FN uint32_t fp_bits(float f)
{
    uint32_t b;
    memcpy(&b, &f, sizeof b);
    return b;
}
BD_FP_FN uint64_t fp_bits(double d)
{
    uint64_t b;
    memcpy(&b, &d, sizeof b);
    return b;
}

BD_FP_FN int fp_clz(uint32_t v)  // v != 0
{
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return __builtin_clz(v);
#endif
}

// (double)f: exponent rebiased by 1023 - 127
BD_FP_FN double widen(float f)
{
    const uint32_t b = fp_bits(f), m = b & 0x7fffffffu;
    uint64_t v = ((uint64_t)m << 29) + (896ull << 52);
    if (m - 0x00800000u >= 0x7f000000u) {  // zero, subnormal, infinity or NaN
        if (m > 0x7f800000u) {
            v = (uint64_t)m << 29 | 0x7ff8ull << 48;
        } else if (m == 0x7f800000u) {
            v = 0x7ff0ull << 48;
        } else if (m == 0) {
            v = 0;
        } else {
            const int s = fp_clz(m) - 8;  // leading bit to position 23
            v = (uint64_t)(897 - s) << 52 | (uint64_t)((m << s) & 0x7fffffu) << 29;
        }
    }
    v |= (uint64_t)(b & 0x80000000u) << 32;
    double d;
    memcpy(&d, &v, sizeof d);
    return d;
}

// (float)d: exponents 897..1150 (a normal float, or infinity by the carry) drop
// 29 bits rounded half to even, by adding half less one and the last bit kept
BD_FP_FN float narrow(double d)
{
    const uint64_t b = fp_bits(d), m = b & 0x7fffffffffffffffull;
    const uint32_t e = (uint32_t)(m >> 52);
    uint32_t v = (uint32_t)((m - (896ull << 52) + 0x0fffffffull + ((m >> 29) & 1u)) >> 29);
    if (e - 897u > 1150u - 897u) {
        if (m > 0x7ff0ull << 48) {
            v = 0x7fc00000u | ((uint32_t)(m >> 29) & 0x7fffffu);
        } else if (e > 1150u) {
            v = 0x7f800000u;
        } else if (e < 873u) {  // below half the smallest subnormal, or zero
            v = 0;
        } else {  // subnormal: units of 2^-149
            const uint64_t M = (m & 0xfffffffffffffull) | 1ull << 52;
            const int s = 926 - (int)e;
            v = (uint32_t)((M + (1ull << (s - 1)) - 1 + ((M >> s) & 1u)) >> s);
        }
    }
    v |= (uint32_t)(b >> 32) & 0x80000000u;
    float f;
    memcpy(&f, &v, sizeof f);
    return f;
}

// no-ops where the precision already is the one asked for
BD_FP_FN double widen(double d) { return d; }
template <class S> BD_FP_FN S narrow_to(double d);
template <> BD_FP_FN double narrow_to<double>(double d) { return d; }
template <> BD_FP_FN float narrow_to<float>(double d) { return narrow(d); }

}  // namespace bd
