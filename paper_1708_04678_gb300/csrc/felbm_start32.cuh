// Start of an FP32 correction of the mass solve: its right-hand side, an FP64 value
// r rounded to a float, and its first iterate s r with s = tau_0 / m, the FP64
// product rounded to a float.  Included by felbm.cu and felbm3d.cu.
#pragma once

#include <cmath>
#include <cstdint>

// The kernels that form them are bound by the FP64 pipe, which runs at 1/64 of the
// FP32 rate and does the conversions too.  So r is split on the integer pipe into
// a float and the 23 bits below it, s into two floats on the host, and the product
// is summed in FP32 to 2^-46 of itself before it is rounded.  Sizes at which a part
// might not be a normal float take the FP64 pipe.  FP64 step (GB300): 2,082,816
// nodes 7.65 ms, with FP64 products and conversions 8.26; on 18,432 nodes, where the
// chain of a thread counts, 155 us, with them 153.
struct Start32 {
    float2 s;                    // s.x + s.y; s.x = 0: out of range
    const double* inv_m;         // 1/m of the node
    double tau0;
    __device__ __forceinline__ void operator()(double r, float& r32, float& first) const {
        const uint32_t h = (uint32_t)__double2hiint(r), l = (uint32_t)__double2loint(r), sign = h & 0x80000000u;
        const uint32_t e = (h & 0x7fffffffu) - (931u << 20);                    // above 2^-92
        if (e < (s.x != 0.0f ? 120u << 20 : 0u)) {
            const uint32_t u = (e + (35u << 20)) << 3 | l >> 29, rem = l & 0x1fffffffu;
            r32 = __uint_as_float(sign | (u + ((rem + 0x0fffffffu + (u & 1u)) >> 29)));   // nearest, ties to even
            const uint32_t below = (u & 0x7f800000u) - (23u << 23);
            const float a = __uint_as_float(u), b = __uint_as_float(below | rem >> 6) - __uint_as_float(below);
            const float p = a * s.x;
            first = __uint_as_float(__float_as_uint(p + fmaf(a, s.y, fmaf(b, s.x, fmaf(a, s.x, -p)))) | sign);
        } else if ((h << 1 | l) == 0u) {
            r32 = first = __uint_as_float(h);
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
