// Correctly rounded FP64 division and square root on the integer pipes.
//
// A GB300 SM issues 2 FP64 operations per clock against 128 integer or FP32
// ones, and a correctly rounded FP64 division or square root built on the
// FP64 pipe holds it for about ten of its slots. These routines use none of
// it: the significand of the result is formed as an integer by schoolbook
// division (two digits of 30 and 23 bits) or digit-by-digit root extraction
// with an FP32 reciprocal as the digit estimate, and rounded from the EXACT
// integer remainder, so the result is the IEEE 754 round-to-nearest value
// whatever the estimate's last bits are (the bounds below leave room for any
// estimate within 2^-21). Operands or results that are zero, subnormal,
// infinite or NaN take the hardware routine.
//
// Measured (GB300, all SMs, independent operations): division 4.1e11/s against
// 6.5e10/s for __ddiv_rn, square root 3.5e11/s against 6.7e10/s for
// __dsqrt_rn. In the FP64 solvers, where both were over half of the FP64
// pipe's time: 32 networks of 5000 nodes x 300 iterations 32.1 -> 21.1 ms, one
// 512-node network x 1000 iterations 29.4 -> 18.8 ms.
//
// The functions are plain integer C but for the FP32 estimate, and compile
// for the host as well, where the tests run them against the host's IEEE
// division and square root with the estimate perturbed.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define F64_FN __device__ __forceinline__
#else
#include <math.h>
#include <string.h>
#define F64_FN static inline
#endif

namespace fe2 {

#ifdef __CUDACC__
F64_FN uint64_t f64_bits(double a) { return (uint64_t)__double_as_longlong(a); }
F64_FN double f64_from(uint64_t b) { return __longlong_as_double((long long)b); }
F64_FN uint32_t f64_mulhi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
// FP32 estimates, read back as integers: rcp of a float given by its bits,
// rsqrt of a float given by its bits (both results are below 2^32)
F64_FN uint32_t f64_est_rcp(uint32_t f) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(f)));
    return min(__float2uint_rz(y), 0x7fffffffu);
}
F64_FN uint32_t f64_est_rsqrt(uint32_t f) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(f)));
    return min(__float2uint_rz(y), 0x7fffffffu);
}
F64_FN double f64_hw_div(double a, double b) { return __ddiv_rn(a, b); }
F64_FN double f64_hw_sqrt(double a) { return __dsqrt_rn(a); }
#else
F64_FN uint64_t f64_bits(double a) { uint64_t b; memcpy(&b, &a, 8); return b; }
F64_FN double f64_from(uint64_t b) { double a; memcpy(&a, &b, 8); return a; }
F64_FN uint32_t f64_mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static int f64_perturb = 0;  // units in the last place added to the FP32 estimates
F64_FN uint32_t f64_est(float y) {
    uint32_t u;
    memcpy(&u, &y, 4);
    u += (uint32_t)f64_perturb;
    memcpy(&y, &u, 4);
    return y < 2147483648.0f ? (uint32_t)y : 0x7fffffffu;
}
F64_FN float f64_f32(uint32_t f) { float x; memcpy(&x, &f, 4); return x; }
F64_FN uint32_t f64_est_rcp(uint32_t f) { return f64_est(1.0f / f64_f32(f)); }
F64_FN uint32_t f64_est_rsqrt(uint32_t f) { return f64_est((float)(1.0 / sqrt((double)f64_f32(f)))); }
F64_FN double f64_hw_div(double a, double b) { return a / b; }
F64_FN double f64_hw_sqrt(double a) { return sqrt(a); }
#endif

constexpr uint64_t kF64Man = 0x000fffffffffffffull, kF64One = 0x0010000000000000ull;

// v = 2^83 / mb - d, 0 <= d < 2.1, for a 53-bit significand mb. The FP32
// estimate v0 of 2^31 / beta, beta = mb / 2^52 in [1, 2), is within a relative
// 2^-21 (truncated operand, approximate reciprocal); one Newton step on
// integers leaves the square of that, and its truncations (beta to 31 bits,
// the product to an integer) move it by -1.1 .. +1, which the final - 1
// turns into a bound from below.
F64_FN uint32_t f64_recip(uint64_t mb) {
    const uint32_t bh = (uint32_t)(mb >> 21);                                          // beta 2^31, truncated
    const uint32_t v0 = f64_est_rcp(0x30000000u | ((uint32_t)(mb >> 29) & 0x7fffffu));  // 2^31 / beta
    const int64_t e = (int64_t)((1ull << 62) - (uint64_t)bh * v0);                     // |e| < 2^42
    const int32_t eh = (int32_t)(e >> 20);                                             // relative error * 2^42
    return (uint32_t)((int32_t)v0 + (int32_t)(((int64_t)(int32_t)v0 * eh) >> 42)) - 1u;
}

// RN(a / b) from v = 2^83 / mb - d for b's significand mb; d < 2.1 as
// f64_recip gives it, or d < 8 with WIDE (f64_sqrt_recip).
//
// With A the numerator's significand, doubled when it is below mb, the
// quotient's significand is A 2^52 / mb in [2^52, 2^53). Digits from v:
//   q1 = A 2^29 / mb, short by d (from v), 0.5 (truncation of A) and 1 (of the
//        product): remainder R1 < 3.6 mb < 2^55, WIDE 9.5 mb < 2^57;
//   q2 = R1 2^23 / mb, short by < 1.1, WIDE < 1.7: R2 < 1.1 mb, WIDE 1.7 mb;
// so the rounded significand is q1 2^23 + q2, plus one when 2 R2 > mb, plus one
// when 2 R2 > 3 mb (WIDE only). (2 R2 = mb never: mb would be a multiple of
// 2^53.) All remainders fit in 64 bits and are exact; the products are taken
// modulo 2^64.
template <bool WIDE>
F64_FN double f64_div_v(double a, double b, uint32_t v) {
    const uint64_t ua = f64_bits(a), ub = f64_bits(b);
    const int ea = (int)(ua >> 52) & 0x7ff, eb = (int)(ub >> 52) & 0x7ff;
    const uint64_t ma = (ua & kF64Man) | kF64One, mb = (ub & kF64Man) | kF64One;
    const bool low = ma < mb;
    const int e = ea - eb + 1022 - (int)low;  // biased exponent - 1
    if ((unsigned)(ea - 1) >= 2046u || (unsigned)(eb - 1) >= 2046u || (unsigned)e >= 2045u)
        return f64_hw_div(a, b);
    const uint64_t A = low ? ma << 1 : ma;
    const uint32_t q1 = f64_mulhi((uint32_t)(A >> 22), v);
    const uint64_t R1 = (A << 29) - (uint64_t)q1 * mb;
    const uint32_t q2 = WIDE ? f64_mulhi((uint32_t)(R1 >> 25), v) >> 3 : f64_mulhi((uint32_t)(R1 >> 24), v) >> 4;
    const uint64_t R2 = ((R1 << 23) - (uint64_t)q2 * mb) << 1;
    const uint64_t Q = ((uint64_t)q1 << 23) + q2 + (R2 > mb) + (WIDE ? (R2 > 3 * mb) : 0);
    return f64_from(((ua ^ ub) & 0x8000000000000000ull) | (((uint64_t)e << 52) + Q));
}

// the reciprocal digit estimate of a divisor, for f64_div_v<false>
F64_FN uint32_t f64_recip_of(double b) { return f64_recip((f64_bits(b) & kF64Man) | kF64One); }

// RN(a / b)
F64_FN double f64_div(double a, double b) { return f64_div_v<false>(a, b, f64_recip_of(b)); }

// RN(sqrt(a)).
//
// m = the significand, doubled for an odd exponent; mu = m / 2^52 in [1, 4).
// The root's significand is the integer nearest to sqrt(m 2^52).
//   v = 2^31 / sqrt(mu) - d, 0 <= d < 8: FP32 estimate, one Newton step, whose
//       truncations move it by -2 .. +6;
//   q1 = 2^29 sqrt(mu), short by < 9.5: remainder R1 = m 2^6 - q1^2 < 2^35;
//   q2 = R1 2^22 / q1: v in the place of 2^60 / q1 and the truncations make it
//       short by < 2.4, the neglected q2^2 / (2 root) long by < 0.6;
// R2 = m 2^52 - Q^2, Q = q1 2^23 + q2, is exact modulo 2^64, and the root
// rounds to Q + k, k = -1 .. 2, where (Q + k - 1/2)^2 < m 2^52 <
// (Q + k + 1/2)^2 (never equal: the square of a half-integer is no integer).
//
// vr receives v: the root's significand is at most 2^53 - 1 (m <= 2^54 - 2), so
// v is also 2^83 / (the root's significand) - d for f64_div_v<true>.
F64_FN double f64_sqrt_recip(double a, uint32_t &vr) {
    const uint64_t ua = f64_bits(a);
    const int ea = (int)(ua >> 52);  // the sign bit makes it >= 2048
    if ((unsigned)(ea - 1) >= 2046u) {
        const double r = f64_hw_sqrt(a);
        vr = f64_recip_of(r);
        return r;
    }
    const int odd = (ea & 1) ^ 1;  // biased exponent even: true exponent odd
    const uint64_t m = ((ua & kF64Man) | kF64One) << odd;
    const int e = (ea - 1023 - odd) >> 1;
    const uint32_t mh = (uint32_t)(m >> 22);  // mu 2^30
    // float mu 2^-62: the estimate is 2^31 / sqrt(mu)
    const uint32_t v0 = f64_est_rsqrt(0x20800000u + (((uint32_t)(odd) << 23) | ((uint32_t)(ua >> 29) & 0x7fffffu)));
    const uint32_t w = f64_mulhi(v0, v0);                             // 2^30 / mu
    const int32_t d = (int32_t)(0x10000000u - f64_mulhi(w, mh));      // 2^28 (1 - mu v0^2)
    const uint32_t v = (uint32_t)((int32_t)v0 + (int32_t)(((int64_t)(int32_t)v0 * d) >> 29)) - 6u;
    vr = v;
    const uint32_t q1 = f64_mulhi(mh, v);                             // 2^29 sqrt(mu)
    const uint64_t R1 = (m << 6) - (uint64_t)q1 * q1;
    const uint32_t q2 = f64_mulhi((uint32_t)(R1 >> 3), v) >> 3;
    const uint64_t Q = ((uint64_t)q1 << 23) + q2;
    const int64_t R2 = (int64_t)((m << 52) - Q * Q);
    const int64_t s = (int64_t)Q;
    const int k = (R2 > -s) + (R2 > s) + (R2 > 3 * s + 2) - 1;
    return f64_from(((uint64_t)(e + 1022) << 52) + Q + (uint64_t)(int64_t)k);
}
F64_FN double f64_sqrt(double a) {
    uint32_t v;
    return f64_sqrt_recip(a, v);
}

}  // namespace fe2
