// fp64_math.cuh -- reciprocal, quotient and logarithm for the FP64 path.  GB300 issues
// two FP64 lanes a clock and SM, so what counts is the number of FP64 instructions:
// exponents, table indices, range checks and conversions are done on the integer pipe.
//   rcp64   Newton-Raphson from an FP32 reciprocal (22 bits, then 44, then 53): 4
//           instructions; within 1 unit in the last place
//   div64   the product with that reciprocal, corrected by its remainder: 7
//   Log64   table-driven (Tang, ACM TOMS 16, 1990): x = 2^k m, m c_i^-1 = 1 + r with
//           |r| < 2^-8, ln x = k ln 2 + ln c_i + log1p(r) by a degree-6 polynomial: 10.
//           Absolute error below 2^-53 max(1, |ln x|) + 2^-54, which is what mu0
//           (ln rho + 1 + ...) needs.
#pragma once

#include <cmath>

#include "df.cuh"

namespace cplbm {

// finite, positive and below FLT_MAX, without an FP64 comparison
__device__ __forceinline__ bool positive64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    return hi < 0x47f00000u && (hi | (unsigned)__double2loint(x)) != 0u;
}

__device__ __forceinline__ double rcp64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    // outside 2^-100 .. 2^100 (or not finite): the correctly rounded function
    if ((hi & 0x7ff00000u) - (923u << 20) >= (200u << 20)) return __drcp_rn(x);
    const float s = __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - 0x38000000u) << 3) |
                                    ((unsigned)__double2loint(x) >> 29));
    const double y = widen(__fdividef(1.0f, s));
    const double z = __fma_rn(y, __fma_rn(-x, y, 1.0), y);
    return __fma_rn(z, __fma_rn(-x, z, 1.0), z);
}
// a / x; rcp: rcp64(x).  Finite a; finite x != 0 (the EOS denominators: 1 - b rho, which is
// zero at the pole alone, and its like).
__device__ __forceinline__ double div64(double a, double x, double rcp) {
    const double q = __dmul_rn(a, rcp);
    return __fma_rn(__fma_rn(-x, q, a), rcp, q);
}
// n / x twice, for densities x down to the smallest subnormal: those whose reciprocal, or
// whose product's remainder, has no place in the type are scaled with their numerators.
__device__ __forceinline__ void quotients64(double& a, double& b, double x) {
    if (((unsigned)__double2hiint(x) & 0x7ff00000u) < (523u << 20)) {
        x = __dmul_rn(x, 0x1p500);
        a = __dmul_rn(a, 0x1p500);
        b = __dmul_rn(b, 0x1p500);
    }
    const double inv = rcp64(x);
    a = div64(a, x, inv);
    b = div64(b, x, inv);
}

struct LogTable {
    static constexpr int kN = 128;
    double2 e[kN];  // 1/c_i and ln c_i, c_i the middle of [1 + i/128, 1 + (i + 1)/128)
};
inline const LogTable& log_table() {  // host
    static const LogTable t = [] {
        LogTable x;
        for (int i = 0; i < LogTable::kN; ++i) {
            x.e[i].x = 1.0 / (1.0 + (i + 0.5) / LogTable::kN);
            x.e[i].y = -std::log(x.e[i].x);
        }
        return x;
    }();
    return t;
}
// logarithm (table in shared memory) and division of the FP64 EOS evaluation
struct Math64 {
    const double2* tab;
    __device__ __forceinline__ double log(double x) const {
        const unsigned hi = (unsigned)__double2hiint(x);
        if (hi - 0x00100000u >= 0x7fe00000u) return ::log(x);  // not positive, normal and finite
        const double2 c = tab[(hi >> 13) & 127u];
        const double m = __hiloint2double((int)((hi & 0x000fffffu) | 0x3ff00000u),
                                          __double2loint(x));
        // the exponent as a double: 2^52 + k + 1023, less 2^52 + 1023
        const double k = __dadd_rn(__hiloint2double(0x43300000, (int)(hi >> 20)),
                                   -(4503599627370496.0 + 1023.0));
        const double r = __fma_rn(m, c.x, -1.0);
        double q = __fma_rn(r, -1.0 / 6.0, 0.2);
        q = __fma_rn(q, r, -0.25);
        q = __fma_rn(q, r, 1.0 / 3.0);
        q = __fma_rn(q, r, -0.5);
        q = __fma_rn(__dmul_rn(r, r), q, r);
        return __dadd_rn(__fma_rn(k, 0.69314718055994530942, c.y), q);
    }
    __device__ __forceinline__ double div(double a, double b) const {
        return div64(a, b, rcp64(b));
    }
    __device__ __forceinline__ bool pos(double x) const {  // x > 0, false for NaN
        const int hi = __double2hiint(x);
        return hi >= 0 && (hi | __double2loint(x)) != 0 &&
               !(hi > 0x7ff00000 || (hi == 0x7ff00000 && __double2loint(x) != 0));
    }
};

}  // namespace cplbm
