// An FP64 value as the nearest double word (hi + lo, FP32): hi = RN24(x),
// lo = RN24(x - hi), by integer arithmetic on the significand.
//
// Conversions to and from FP64 run at 2 per cycle and SM, and the direct form takes
// three of them and an FP64 subtraction a value, which bounded the field conversions
// of the reliable updates (one-flavour field at 24^3x48 59 -> 18 us).  Here the 53-bit
// significand is cut at FP32's last place, rounded to nearest even by the
// 29 bits below, and those bits less the rounding, a signed integer, are converted
// and scaled exactly.  Values whose parts are not all normal FP32 numbers (zeros,
// exponents below -74 or above 126, infinities, NaN) take the direct form.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define TM_HD __host__ __device__ __forceinline__
#else
#define TM_HD inline
#endif

namespace tmk {

struct SplitPair {
    float h, l;
};
// (out of line: predicated, its conversions would issue for every value)
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
inline SplitPair df_split_direct(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}

TM_HD void df_split(double x, float& h, float& l) {
    uint64_t b;
    memcpy(&b, &x, 8);
    const uint32_t top = (uint32_t)(b >> 32);
    const int e = (int)((top >> 20) & 0x7ff) - 1023;
    if (e < -74 || e > 126) {
        const SplitPair p = df_split_direct(x);
        h = p.h;
        l = p.l;
        return;
    }
    const uint32_t rest = (uint32_t)b & 0x1fffffffu;             // the 29 bits below FP32's significand
    uint32_t hb = (uint32_t)(e + 127) << 23 | (uint32_t)(b >> 29 & 0x7fffffu);
    const uint32_t up = rest > 0x10000000u || (rest == 0x10000000u && (hb & 1u)) ? 1u : 0u;
    hb += up;                                                   // (a carry moves to the exponent)
    int d = (int)rest - (int)(up << 29);                        // (x - hi) / 2^(e - 52), up to the sign
    const uint32_t sign = top & 0x80000000u;
    if (sign) d = -d;
    hb |= sign;
    const uint32_t sb = (uint32_t)(e - 52 + 127) << 23;
    float scale;
    memcpy(&h, &hb, 4);
    memcpy(&scale, &sb, 4);
    l = (float)d * scale;
}

}  // namespace tmk
