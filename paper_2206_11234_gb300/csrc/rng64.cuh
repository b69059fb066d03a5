// Binary64 Box–Muller of the reference stepper and of its probe: u0 = (w + 1/2)
// 2^-32 from a radius word, u1 = (h + 1/2) 2^-16 from a 16-bit angle field,
// r = sqrt(-2 ln u0), (r cos 2 pi u1, r sin 2 pi u1).
//
// GB300 issues one binary64 warp instruction per SM every 16 cycles, so the
// binary64 instructions are all that counts.  With the library's log, sqrt and
// sincos a pair took about 70 of them; here it takes 13, everything else being
// integer work and two 16-byte table reads:
//   * the 2^16 angles 2 pi u1 (the binary64 product) have their correctly rounded
//     cosines and sines in a table of 1 MB, which stays in the L2 cache;
//   * u0 has 33 significant bits.  With u0 = 2^-n m / 2, m in [1, 2), and an entry
//     inv ~ 1/m of 20 bits chosen by the top 10 bits of m, r' = 2 - 2 m inv is exact
//     and |r'| <= 2^-10 (table-driven logarithm, Tang, ACM TOMS 16 (1990)):
//     -2 ln u0 = n 2 ln 2 + 2 ln(2 inv) - 2 ln(1 - r'/2), the last term as its series
//     to r'^5.  Near u0 = 1 the entry is 1/2 and both constants vanish, so the
//     result keeps its relative accuracy there;
//   * the root and the reciprocal by one third-order step from the hardware's seeds:
//     Householder's iteration of the second order (Householder, The Numerical
//     Treatment of a Single Nonlinear Equation (1970)), for 1/x the geometric series
//     of 1/(1 - e) to e^2, for the root the binomial series of (1 - e)^(-1/2) to e^2.
// Against 80-bit arithmetic of the same angles the radius errs by 5.2e-17 on
// average and 2.9e-16 at most, the cosine by half a unit in the last place.
// The tables are written at build time (build.py) in exact integer arithmetic.
//
// A translation unit without binary64 kernels defines FPT_NO_F64 first, which keeps
// the tables out: 1 MB of device memory per unit, and 5 ms of its first call.
#pragma once
#include <cstdint>

#ifndef FPT_NO_F64
#include "f64_tables.inc"  // bits of kTrig64[65536] {cos, sin}, kLog64[1024] {-2 inv, 2 ln(2 inv)}, kLn2N64[33] = n 2 ln 2
#endif
#include "rng.cuh"

namespace fpt {

struct PairF64 {
    double r, c, s;  // normals r c, r s
};

#ifdef FPT_NO_F64
__device__ PairF64 pair_f64(uint32_t rad, uint32_t h);
__device__ PairF64 group_pair_f64(const uint32_t V[12], int j, int p);
#endif

__device__ __forceinline__ double2 table_pair(const ulonglong2* t) {
    const ulonglong2 v = __ldg(t);
    return make_double2(__longlong_as_double((long long)v.x), __longlong_as_double((long long)v.y));
}

// y to about 2^-20, by the reciprocal (square root) unit
__device__ __forceinline__ double rcp_seed(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}

// 1/x by one third-order step y (1 + e + e^2), e = 1 - x y
__device__ __forceinline__ double reciprocal(double x) {
    const double y = rcp_seed(x);
    const double e = __fma_rn(-x, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}

// sqrt(L) by one third-order step g (1 + e/2 + 3 e^2/8), g = L y, e = 1 - g y
__device__ __forceinline__ double root(double L) {
    const double y = rsqrt_seed(L);
    const double g = __dmul_rn(L, y);
    const double e = __fma_rn(-g, y, 1.0);
    return __fma_rn(__dmul_rn(g, e), __fma_rn(e, 0.375, 0.5), g);
}

#ifndef FPT_NO_F64
// -2 ln((w + 1/2) 2^-32)
__device__ __forceinline__ double minus_two_ln(uint32_t w) {
    const uint64_t U = 2ull * w + 1ull;  // u0 = U 2^-33
    const int lead = __clzll((long long)U);
    const uint64_t bits = (U << lead) << 1;  // the fraction of m, left aligned
    const double m = __longlong_as_double((long long)(0x3ff0000000000000ull | (bits >> 12)));
    const double2 t = table_pair(&kLog64[(int)(bits >> 54)]);
    const double base = __dadd_rn(t.y, __longlong_as_double((long long)__ldg(&kLn2N64[lead - 31])));
    const double x = __fma_rn(m, t.x, 2.0);
    double q = __fma_rn(x, 1.0 / 80.0, 1.0 / 32.0);
    q = __fma_rn(q, x, 1.0 / 12.0);
    q = __fma_rn(q, x, 0.25);
    return __dadd_rn(base, __fma_rn(__dmul_rn(x, x), q, x));
}

__device__ __forceinline__ PairF64 pair_f64(uint32_t rad, uint32_t h) {
    const double2 t = table_pair(&kTrig64[h & 0xffffu]);
    return PairF64{root(minus_two_ln(rad)), t.x, t.y};
}

// pair p of block j of a 16-step group's words
__device__ __forceinline__ PairF64 group_pair_f64(const uint32_t V[12], int j, int p) {
    const uint32_t ang = V[3 * j + 2];
    return pair_f64(V[3 * j + p], p == 0 ? ang >> 16 : ang & 0xffffu);
}

// The four normals of 4-step block k as values.
__device__ __forceinline__ void normals4_f64(const PhiloxLane& l, uint32_t k, const PhiloxKeys& K, double xi[4]) {
    const BlockWords w = block_words(l, k, K);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const PairF64 q = pair_f64(p == 0 ? w.rad0 : w.rad1, p == 0 ? w.ang >> 16 : w.ang & 0xffffu);
        xi[2 * p] = __dmul_rn(q.r, q.c);
        xi[2 * p + 1] = __dmul_rn(q.r, q.s);
    }
}

#endif  // FPT_NO_F64

}  // namespace fpt
