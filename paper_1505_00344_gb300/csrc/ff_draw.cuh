// ff_draw.cuh -- uniform draws from a group's box (paper Appendix A, "Particle
// Group"), shared by the seeding kernel and the integrator's in-kernel reset.
//
// A draw is the top 24 bits k of a SplitMix64 output (Steele, Lea & Flood 2014:
// output n of the stream seeded with s is the variant-13 finaliser of
// s + n * 0x9E3779B97F4A7C15), u = k / 2^24, and x = lo + width * u in double, each
// operation rounded, then rounded to float.
//
// The FP64 pipe runs 2 lanes per clock and SM here, and its five operations per value
// bound the seeding: 122 us for the 12.6M values of 4,194,304 Lorenz particles, whose
// 50 MB take 8 us to write.  So the value is formed in pairs of floats, with an error
// bound that decides whether its rounding to float is certain; where it is not, the double
// formula runs.  A box of short bounds (-30..30: multiples of 2, k / 2^24 of its width
// multiples of 2^-22) has values halfway between floats one time in eight, which no nonzero
// bound could decide, but its pair arithmetic is exact; of other boxes about one value in 2^11
// takes the double formula.  Every result is the double formula's: 122 us -> 29 us.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace ff {

constexpr uint64_t kSplitMixGamma = 0x9E3779B97F4A7C15ULL;

// The variant-13 finaliser: output n of the stream seeded with s is splitmix64_mix(s + n * gamma).
__device__ __forceinline__ uint64_t splitmix64_mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// One variable's interval: the double formula's operands, and lo and width / 2^24 as
// unevaluated sums of two floats.
struct DrawBox {
    double lo, width;
    float lh, ll, wh, wl;
    float tol;  // bound on the pair arithmetic's error; NaN: the double formula always
    float pad_;
};

// The lowest set bit of x as a power of two (infinity for 0).
inline double draw_low_bit(double x) {
    if (x == 0.0) return INFINITY;
    int e = 0;
    uint64_t m = (uint64_t)std::ldexp(std::fabs(std::frexp(x, &e)), 53);  // 53-bit integer
    for (e -= 53; (m & 1u) == 0; m >>= 1) ++e;
    return std::ldexp(1.0, e);
}

// tol: 0 where lo and width are floats whose values all lie on a grid g with |lo| + |width| <=
// 2^45 g: the product's two parts, the sum and its error and t are then exact (t's terms are
// multiples of g below 2^24 g), as are the double formula's operations.  Otherwise the pair
// arithmetic's error relative to |lo| + |width|: lo and width to 2^-48 each, the roundings of
// the low parts 2^-48 + 2^-46 + 2 * 2^-47, of t +- tol 2^-46, and the double formula's own
// roundings 2^-52; 2^-43 leaves a factor of two.  Scales outside [2^-40, 2^100] could lose
// low parts to underflow or overflow and take the double formula.
inline DrawBox draw_box(double lo, double hi) {
    DrawBox b{};
    b.lo = lo;
    b.width = hi - lo;
    const double scale = std::fabs(lo) + std::fabs(b.width);
    b.tol = NAN;
    if (scale >= 0x1p-40 && scale <= 0x1p100) {
        const double w = b.width * 0x1p-24;  // exact but for a width whose part in x is far below tol
        b.lh = (float)lo;
        b.ll = (float)(lo - (double)b.lh);
        b.wh = (float)w;
        b.wl = (float)(w - (double)b.wh);
        const double grid = std::fmin(draw_low_bit(lo), draw_low_bit(w));
        b.tol = (b.ll == 0.0f && b.wl == 0.0f && scale <= 0x1p45 * grid) ? 0.0f : (float)(scale * 0x1p-43);
    }
    return b;
}

// The double formula.  A call, not inlined: inlined, the toolchain predicates it, and the
// predicated-off instructions still took their turns on the FP64 pipe (no change in time).
static __device__ __noinline__ float draw_double(uint32_t k, double lo, double width) {
    const double u = (double)k * (1.0 / 16777216.0);
    return __double2float_rn(__dadd_rn(lo, __dmul_rn(width, u)));
}

// The value of a draw whose finaliser output is z.
__device__ __forceinline__ float draw_value(uint64_t z, const DrawBox& b) {
    const float k = (float)(uint32_t)(z >> 40);  // 24 bits: exact
    const float ph = __fmul_rn(k, b.wh);
    const float pl = fmaf(k, b.wl, fmaf(k, b.wh, -ph));  // k * width / 2^24 = ph + pl
    const float s = __fadd_rn(b.lh, ph);                 // lh + ph = s + e exactly (Knuth's two-sum)
    const float v = __fsub_rn(s, b.lh);
    const float e = __fadd_rn(__fsub_rn(b.lh, __fsub_rn(s, v)), __fsub_rn(ph, v));
    const float t = __fadd_rn(e, __fadd_rn(b.ll, pl));
    // rounding is monotone: where both ends of the error interval round to the same float,
    // so does the double formula's value inside it
    const float up = __fadd_rn(s, __fadd_rn(t, b.tol)), down = __fadd_rn(s, __fsub_rn(t, b.tol));
    return up == down ? up : draw_double((uint32_t)(z >> 40), b.lo, b.width);
}

}  // namespace ff
