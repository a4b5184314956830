// Fixed-point arithmetic for the FP64 fields.
//
// GB300 issues one FP64 FMA per warp and SM sub-partition every 80 cycles,
// conversions between FP64 and other types at the same rate, but one 32 x 32
// -> 64-bit integer multiply-add (IMAD.WIDE) every 4 cycles (measured).  The entries of SU(3) matrices are bounded by 1,
// so a real can be held as a 64-bit integer X with value X 2^-60, and a
// product of two of them summed in three such multiply-adds: with
// X = h 2^32 + l (l signed, |l| < 2^31),
//   X Y 2^-64 = h_x h_y + (h_x l_y + l_x h_y) 2^-32 + l_x l_y 2^-64,
// the first term and the middle sum in 64-bit accumulators of their own; the
// last term is dropped (below 2^-58 per product, 2^-59.6 rms).  A 3 x 3
// complex product takes ~1 600 cycles per warp this way (324 multiply-adds and
// ~160 additions, shifts and splits, bound by the multiplier; measured, the
// same for 2 to 4 blocks of 128 per SM) against 8 640 of FP64 FMAs, and its
// absolute error is about 2^-58 where the FP64 chain of six FMAs leaves
// 2^-54.6 rms: results are closer to the exact ones than FP64's.  Tried and
// not faster: accumulators interleaved across a row (1 594, or 1 690 when the
// order is pinned), a three-multiplication complex product (243 multiply-adds
// but ~400 other operations: 2 000).
//
// Bounds.  For rows of norm at most 1 (SU(3) to the 1e-6 of the input check)
// a dot product of length 6 stays below 6 2^56 in the high accumulator and,
// by Cauchy-Schwarz, below 2 sqrt(6) 2^59 < 2^62 in the middle one.  Values up
// to 8 in magnitude are representable; every kernel states its operand bounds.
//
// The functions are plain integer code, compiled for the host as well (the
// host tests run them).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mcg {

#define MCG_HD __host__ __device__ __forceinline__

struct fx {  // value (h 2^32 + l) 2^-60
    int h, l;
};
struct alignas(16) cfx {
    fx re, im;
};
struct facc {  // value hi 2^-56 + mid 2^-88
    long long hi, mid;
};

// X as (h, l).  l = -2^31 is moved up by one unit, so that (-h, -l) is the
// negation of every value (and the smearing step measured 10 % faster with the
// extra minimum than without).
MCG_HD fx fx_split(long long X) {
    fx r;
    r.l = (int)X;
    r.h = (int)(X >> 32) - (r.l >> 31);
    r.l = r.l < -0x7fffffff ? -0x7fffffff : r.l;
    return r;
}
MCG_HD long long fx_join(fx a) { return ((long long)a.h << 32) + a.l; }
MCG_HD fx fx_neg(fx a) {
    fx r;
    r.h = -a.h;
    r.l = -a.l;
    return r;
}
MCG_HD facc facc_zero() {
    facc s;
    s.hi = s.mid = 0;
    return s;
}
MCG_HD void fx_mac(facc& s, fx a, fx b) {
    s.hi += (long long)a.h * b.h;
    s.mid += (long long)a.h * b.l;
    s.mid += (long long)a.l * b.h;
}
MCG_HD void fx_msc(facc& s, fx a, fx b) {  // s - a b
    s.hi += (long long)(-a.h) * b.h;
    s.mid += (long long)(-a.h) * b.l;
    s.mid += (long long)a.l * (-b.h);
}
MCG_HD long long facc_get(facc s) { return (long long)((unsigned long long)s.hi << 4) + (s.mid >> 28); }
MCG_HD long long fx_mul(fx a, fx b) {
    facc s = facc_zero();
    fx_mac(s, a, b);
    return facc_get(s);
}

// ---- FP64 <-> fixed point by integer operations ------------------------------
// |d| < 8; bits below 2^-60 are dropped.  (Values outside, infinities and NaN
// give some in-range integer: the callers keep them out.)
MCG_HD long long fx_from_bits(unsigned long long bits) {
    const unsigned hi = (unsigned)(bits >> 32);
    const int r = 1025 - (int)((hi >> 20) & 0x7ff);  // right shift of mantissa 2^10
    const unsigned long long m = ((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
    const unsigned long long v = r > 63 ? 0ULL : m >> (r & 63);
    const long long sg = (long long)bits >> 63;
    return ((long long)v ^ sg) - sg;
}
// X 2^-60 rounded to FP64 (ties away from zero)
MCG_HD unsigned long long fx_to_bits(long long X) {
    const long long sg = X >> 63;
    unsigned long long m = (unsigned long long)((X ^ sg) - sg);
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)m);
#else
    const int z = m ? __builtin_clzll(m) : 64;
#endif
    // top bit to 62; the value is then m 2^(-60 - (z - 1))
    m = z > 0 ? m << ((z - 1) & 63) : m >> 1;
    const unsigned long long q = (m + (1ULL << 9)) >> 10;  // 53 bits, implicit one at bit 52
    // exponent field: 1023 + 2 - (z - 1), less the one the implicit bit adds
    const unsigned long long d = q + ((unsigned long long)(1025 - z) << 52);
    const unsigned long long s = (unsigned long long)sg & 0x8000000000000000ULL;
    return X == 0 ? 0ULL : (d | s);
}

#ifdef __CUDACC__
__device__ __forceinline__ fx fx_of(double d) { return fx_split(fx_from_bits((unsigned long long)__double_as_longlong(d))); }
__device__ __forceinline__ double fx_double(long long X) { return __longlong_as_double((long long)fx_to_bits(X)); }
#endif

#ifdef __CUDACC__
// A matrix (entry (r, k) at src[r sr + k sc]) the fixed-point sweep does not
// take: an entry above 1.03 in magnitude or not finite, or a row whose squared
// norm is off 1 by 5 % (tiny rows would lose relative precision).
__device__ __forceinline__ bool fx_bad_matrix(const double2* src, size_t sr, size_t sc) {
    bool bad = false;
#pragma unroll 1
    for (int r = 0; r < 3; ++r) {
        float n2 = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double2 d = src[r * sr + k * sc];
            bad = bad || (__double2hiint(d.x) & 0x7fffffff) > 0x3ff07ae1 || (__double2hiint(d.y) & 0x7fffffff) > 0x3ff07ae1;
            const float x = (float)fx_of(d.x).h, y = (float)fx_of(d.y).h;  // unit 2^-28
            n2 = fmaf(x, x, fmaf(y, y, n2));
        }
        bad = bad || !(fabsf(n2 * 0x1p-56f - 1.f) < 0.05f);
    }
    return bad;
}
#endif

// ---- 3 x 3 complex matrices (row-major) ---------------------------------------
MCG_HD void cfx_mac(facc& re, facc& im, cfx a, cfx b) {
    fx_mac(re, a.re, b.re);
    fx_msc(re, a.im, b.im);
    fx_mac(im, a.re, b.im);
    fx_mac(im, a.im, b.re);
}
// a conj(b)
MCG_HD void cfx_macc(facc& re, facc& im, cfx a, cfx b) {
    fx_mac(re, a.re, b.re);
    fx_mac(re, a.im, b.im);
    fx_mac(im, a.im, b.re);
    fx_msc(im, a.re, b.im);
}
MCG_HD cfx cfx_get(facc re, facc im) {
    cfx r;
    r.re = fx_split(facc_get(re));
    r.im = fx_split(facc_get(im));
    return r;
}
// Row of a b (DAG: of a b^dag) to t, a its row of the left factor.
template <bool DAG>
MCG_HD void m3fx_row(const cfx* a, const cfx* b, cfx* t) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        facc x = facc_zero(), y = facc_zero();
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (DAG)
                cfx_macc(x, y, a[k], b[3 * j + k]);
            else
                cfx_mac(x, y, a[k], b[3 * k + j]);
        }
        t[j] = cfx_get(x, y);
    }
}
// a <- a b (DAG: a b^dag)
template <bool DAG>
MCG_HD void m3fx_mul_inplace(cfx* a, const cfx* b) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        cfx t[3];
        m3fx_row<DAG>(a + 3 * i, b, t);
#pragma unroll
        for (int j = 0; j < 3; ++j) a[3 * i + j] = t[j];
    }
}

}  // namespace mcg
