// Start of an FP32 correction of the mass solve: its right-hand side, an FP64 value
// r rounded to a float, and its first iterate s r with s = tau_0 / m, the FP64
// product rounded to a float.  Included by felbm.cu and felbm3d.cu.
#pragma once

#include <cmath>
#include <cstdint>

// The kernels that form them are bound by the FP64 pipe, which runs at 1/64 of the
// FP32 rate and does the conversions too.  So r is split on the integer pipe into
// a float and the 23 bits below it, s into two floats on the host, and the product
// is summed in FP32 to 2^-46 of itself before it is rounded.  Small values, which
// the tails of an interface are full of, are scaled by 2^64 for it, and those
// whose float and product are zero are zero; what is left (between them, large or
// not finite) takes the FP64 pipe.  FP64 step (GB300): 2,082,816 nodes 7.62 ms, with
// FP64 products and conversions 8.26; 8,320 nodes 90.3 us, with the small values on
// the FP64 pipe 93.5.
struct Start32 {
    float2 s;                    // s.x + s.y; s.x = 0: out of range
    const double* inv_m;         // 1/m of the node
    double tau0;
    __device__ __forceinline__ void operator()(double r, float& r32, float& first) const {
        const uint32_t h = (uint32_t)__double2hiint(r), l = (uint32_t)__double2loint(r), sign = h & 0x80000000u, x = h ^ sign;
        // r and s r below 2^-150 (s.x < 2^(its exponent + 1)), 2^-116 <= r < 2^28
        const bool none = x < (871u - (max(__float_as_uint(s.x) >> 23, 127u) - 127u)) << 20;
        if (s.x != 0.0f && (none || x - (907u << 20) < 144u << 20)) {
            const bool small = x < 931u << 20;                                      // 2^-92
            const uint32_t e = none ? 35u << 20 : x - ((small ? 832u : 896u) << 20);
            const uint32_t u = e << 3 | l >> 29, rem = l & 0x1fffffffu;
            const uint32_t near = u + ((rem + 0x0fffffffu + (u & 1u)) >> 29);       // nearest, ties to even
            const uint32_t below = (u & 0x7f800000u) - (23u << 23);
            const float a = __uint_as_float(u), b = __uint_as_float(below | rem >> 6) - __uint_as_float(below);
            const float p = a * s.x, scale = __uint_as_float(sign | (none ? 0u : small ? 63u << 23 : 127u << 23));
            r32 = __uint_as_float(near) * scale;
            first = (p + fmaf(a, s.y, fmaf(b, s.x, fmaf(a, s.x, -p)))) * scale;
        } else {
            r32 = (float)r;
            first = (float)(r * (*inv_m * tau0));
        }
    }
};

// s in two floats (host).
inline float2 split_scale(double s) {
    const float hi = (float)s, lo = (float)(s - (double)hi);
    return std::isfinite(hi) && hi > 0x1p-10f && hi < 0x1p60f ? make_float2(hi, lo) : make_float2(0.0f, 0.0f);
}
