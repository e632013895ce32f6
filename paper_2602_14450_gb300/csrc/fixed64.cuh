// Fixed-point arithmetic of the FP64 hopping term (hop64_impl.cuh).
//
// GB300 executes 2 FP64 fused multiply-adds per cycle and SM (1.06 TFLOP/s
// measured, 1/70 of FP32), and 32 x 32 + 64-bit integer multiply-adds about 14
// times as fast. The hop is a sum of products of SU(3) link entries (at most 1
// in size) with neighbour spinors of one scale, so it is formed in 64-bit
// fixed point, three integer multiply-adds for one FP64 one:
//
//   link     u = 2^-61 (u1 2^32 + u0)                     signed 32-bit digits u1, u0
//   spinor   p = 2^(E-1081) * (a 60-bit integer)           E: largest biased exponent of a neighbour so far (acc is
//                                                          shifted when a later one exceeds it)
//   half spinor h = p +- p' = 2^(E-1081) (h1 2^32 + h0)
//   u h      = 2^(E-1078) (u1 h1 + (u1 h0 + u0 h1) 2^-32)  (u0 h0 is below the last unit)
//   H        = 2^(E-1078) * (64-bit sum over the eight directions)
//
// Errors, in units of 2^(E-1078), at most 2^-55 of the largest neighbour real:
// a product of a link row with a column is off by at most 2.8 (spinor reals cut
// at 1/8 each: 0.6; u0 h0 left out: 1.5; link entries: 0.2; its own rounding:
// 0.5), of a t hop, doubled, by 4.8; six of the first and one of the second
// make 21.6 per real of the sum, shifts of the sum less than 2 more. Then the
// sum is rounded once to FP64.
//
// These errors go with the largest neighbour of the site, those of FP64
// arithmetic with each real by itself: 14 x 2^-53 times the sum S of the sizes
// of its products (a rounding of the projection, six of the colour row, seven
// of the sum). So a real may be formed here when S >= 1.69 x 2^53 units, where
// 14 x 2^-53 S is 23.6 units. hop64_kernel sums the products of the entries' sizes
// rounded down, links to 2^-5 and half spinors to 2^(E-1027), which S is never
// below; SIZE_MIN is that in its units of 2^(E-1032). On rough links 1 site in
// 10^6 fails; components fed by small spinor parts or small link entries alone do,
// and reals that are zero.
// The relative error of a hop of Gaussian fields is 0.50e-16 against 1.42e-16
// in FP64 arithmetic (tests/test_gpu_fixed64_exact.py), of D_W, with its
// epilogue in FP64, 0.92e-16 against 1.0e-16.
//
// Bounds (rows of unit norm, |h| < 2^60): |sum u1 h0| <= sqrt(6) 2^29 2^31 and
// |sum u0 h1| <= 6 2^31 2^28, together 6.3e18 < 2^63; a product is at most
// sqrt(6) 2^60 / 8, and 6 + 2 / 2 of them stay below 2^61.2.
#pragma once

#include <math.h>
#include <string.h>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace wd {
namespace fx {

// Neighbours whose largest biased exponent lies outside [E_MIN, E_MAX] (and are not zero) take the FP64 path of
// the site: below, the result could be subnormal; above, it could overflow or the input is not finite.
constexpr int E_MIN = 70, E_MAX = 2030;
// The least size of a real's products, in units of 2^(E-1032), at which fixed point is as exact as FP64 arithmetic
// (above). Their sum stays below 2^16: 6 x 32 x 64 sqrt(6) + 2 x 32 x 32 sqrt(6).
constexpr unsigned SIZE_MIN = 216;

// v >> s, zero for s >= 64.
__host__ __device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned s) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s > 63 ? 0ull : v >> s;
#endif
}

// The 64-bit fixed-point link entry of a double in [-1.001, 1.001] as (u0, u1): both digits may be negated.
__host__ __device__ __forceinline__ void link_digits(double u, int& u0, int& u1) {
    const double s = u * 2305843009213693952.0;   // 2^61
#ifdef __CUDA_ARCH__
    long long v = __double2ll_rn(s);
#else
    long long v = llrint(s);
#endif
    int lo = (int)(unsigned)(unsigned long long)v;
    if (lo == (int)0x80000000) {                  // -2^31 has no negative: move the entry by one unit
        v += 1;
        lo += 1;
    }
    u0 = lo;
    u1 = (int)((v - lo) >> 32);
}
__host__ __device__ __forceinline__ double link_value(int u0, int u1) {
    return ((double)u1 * 4294967296.0 + (double)u0) * (1.0 / 2305843009213693952.0);
}

// A real (high and low word of its FP64 value) in units of 2^(E-1081), E >= its biased exponent: the value is
// v - neg with v the one's complement of the magnitude when neg = -1.
struct Fixed {
    unsigned long long v;
    int neg;
};
__host__ __device__ __forceinline__ Fixed fixed(unsigned hi, unsigned lo, int E) {
    const unsigned mh = ((hi << 11) | (lo >> 21)) | 0x80000000u;   // the significand, leading bit at the top
    const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 11);
    // 5 + E - exponent, from the difference of the exponent fields (the fraction below cannot borrow)
    const unsigned s = ((((unsigned)(5 + E) << 20) | 0xFFFFFu) - (hi & 0x7FFFFFFFu)) >> 20;
    Fixed f;
    f.neg = (int)hi >> 31;
    f.v = shr64(m, s) ^ (unsigned long long)(long long)f.neg;
    return f;
}
// a, or its negative for mask = -1.
__host__ __device__ __forceinline__ Fixed signed_by(Fixed a, int mask) {
    a.v ^= (unsigned long long)(long long)mask;
    a.neg ^= mask;
    return a;
}
__host__ __device__ __forceinline__ long long sum(Fixed a, Fixed b) {
    return (long long)(a.v + b.v + (unsigned)-(a.neg + b.neg));
}

// Signed 32-bit digits of a 61-bit integer.
__host__ __device__ __forceinline__ void digits(long long h, int& h0, int& h1) {
    h0 = (int)(unsigned)(unsigned long long)h;
    h1 = (int)(h >> 32) + (int)((unsigned)h0 >> 31);
#ifdef __CUDA_ARCH__
    // hides where the digits come from: seen as parts of h, their products become 64-bit multiplications of
    // three instructions instead of one wide multiply-add
    asm("" : "+r"(h0), "+r"(h1));
#endif
}

// One complex entry of U h, (sum_b U_ab h_b) in units of 2^(E-1078): u0, u1 the digits of a link row
// (re, im of b = 0..2), n0, n1 those of minus its imaginary parts, h0, h1 the digits of one column.
__host__ __device__ __forceinline__ void row_mul(const int (&u0)[6], const int (&u1)[6], const int (&n0)[3],
                                                 const int (&n1)[3], const int* h0, const int* h1, long long& re,
                                                 long long& im) {
    long long mr = 1ll << 31, mi = 1ll << 31, hr = 0, hi = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int x0 = h0[2 * b], x1 = h1[2 * b], y0 = h0[2 * b + 1], y1 = h1[2 * b + 1];
        hr += (long long)u1[2 * b] * x1;
        hr += (long long)n1[b] * y1;
        hi += (long long)u1[2 * b] * y1;
        hi += (long long)u1[2 * b + 1] * x1;
        mr += (long long)u1[2 * b] * x0;
        mr += (long long)u0[2 * b] * x1;
        mr += (long long)n1[b] * y0;
        mr += (long long)n0[b] * y1;
        mi += (long long)u1[2 * b] * y0;
        mi += (long long)u0[2 * b] * y1;
        mi += (long long)u1[2 * b + 1] * x0;
        mi += (long long)u0[2 * b + 1] * x1;
    }
    re = hr + (int)(mr >> 32);
    im = hi + (int)(mi >> 32);
}

// The double nearest to x * 2^(E-1078), E in [E_MIN, E_MAX]: x is put together from its words with one rounding
// (2^84 + 2^32 hi, hi offset by 2^31, and 2^52 + lo are exact doubles), and the scale goes into the exponent field.
__host__ __device__ __forceinline__ double to_double(long long x, int E) {
    const unsigned lo = (unsigned)(unsigned long long)x, hi = (unsigned)((unsigned long long)x >> 32) ^ 0x80000000u;
#ifdef __CUDA_ARCH__
    const double a = __hiloint2double(0x45300000, (int)hi), b = __hiloint2double(0x43300000, (int)lo);
    const double d = __dadd_rn(__dadd_rn(a, -19342822341709703277445120.0), b);
    const int top = __double2hiint(d);
    return __hiloint2double(top ? top + ((E - 1078) << 20) : 0, __double2loint(d));
#else
    const double d = (double)x;
    (void)lo;
    (void)hi;
    return d == 0.0 ? 0.0 : ldexp(d, E - 1078);
#endif
}

}  // namespace fx
}  // namespace wd
