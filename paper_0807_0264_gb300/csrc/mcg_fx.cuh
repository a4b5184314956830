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
// The unit is absolute: an entry far below 1 keeps its digits down to 2^-60 (2^-58 in
// the sweep) only, where FP64 keeps 53 bits of any size.  That matters to fields of
// which every link is near the identity (1e-8 from it: eight digits fewer of the
// distance), not to entries of order one.
//
// The functions are plain integer code, compiled for the host as well (the
// host tests run them).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mcg_common.cuh"

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
// X 2^-60 rounded to FP64 (ties away from zero; half = 511: towards zero)
MCG_HD unsigned long long fx_to_bits(long long X, unsigned half = 512) {
    const long long sg = X >> 63;
    unsigned long long m = (unsigned long long)((X ^ sg) - sg);
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)m);
#else
    const int z = m ? __builtin_clzll(m) : 64;
#endif
    // top bit to 62; the value is then m 2^(-60 - (z - 1))
    m = z > 0 ? m << ((z - 1) & 63) : m >> 1;
    const unsigned long long q = (m + half) >> 10;  // 53 bits, implicit one at bit 52
    // exponent field: 1023 + 2 - (z - 1), less the one the implicit bit adds
    const unsigned long long d = q + ((unsigned long long)(1025 - z) << 52);
    const unsigned long long s = (unsigned long long)sg & 0x8000000000000000ULL;
    return X == 0 ? 0ULL : (d | s);
}

#ifdef __CUDACC__
__device__ __forceinline__ fx fx_of(double d) { return fx_split(fx_from_bits((unsigned long long)__double_as_longlong(d))); }
__device__ __forceinline__ double fx_double(long long X) { return __longlong_as_double((long long)fx_to_bits(X)); }
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

// ---- near-unitary matrices: re-unitarisation -----------------------------------
// 1 / sqrt(1 + d) - 1 for |d| < 2^-12, both in units of 2^-60: the binomial series
// to d^4 (the next term is below 2^-62)
MCG_HD long long fx_rsqrt1(long long d) {
    const fx s = fx_split(d);
    long long e = fx_mul(s, fx_split(35LL << 53)) - (5LL << 56);
    e = fx_mul(s, fx_split(e)) + (3LL << 57);
    e = fx_mul(s, fx_split(e)) - (1LL << 59);
    return fx_mul(s, fx_split(e));
}
MCG_HD long long fx_row_norm2(const cfx* r) {
    facc n = facc_zero();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        fx_mac(n, r[k].re, r[k].re);
        fx_mac(n, r[k].im, r[k].im);
    }
    return facc_get(n);
}
MCG_HD void fx_scale_row(cfx* r, long long e) {  // r += e r
    const fx s = fx_split(e);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r[k].re = fx_split(fx_join(r[k].re) + fx_mul(s, r[k].re));
        r[k].im = fx_split(fx_join(r[k].im) + fx_mul(s, r[k].im));
    }
}
MCG_HD bool fx_far(long long d) { return d > (1LL << 48) || d < -(1LL << 48); }
// Row 0 normalised, row 1 orthogonalised and normalised, row 2 = conj(row0 x
// row1), as m3_reunitarise.  True (and m undefined) when a norm is off 1 by more
// than 2^-12: the caller takes the FP64 form.
MCG_HD bool m3fx_reunitarise(cfx* m) {
    const long long one = 1LL << 60, d0 = fx_row_norm2(m) - one;
    fx_scale_row(m, fx_rsqrt1(d0));
    facc px = facc_zero(), py = facc_zero();  // conj(r0) . r1
#pragma unroll
    for (int k = 0; k < 3; ++k) cfx_macc(px, py, m[3 + k], m[k]);
    const fx qx = fx_split(facc_get(px)), qy = fx_split(facc_get(py));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        facc x = facc_zero(), y = facc_zero();
        cfx p;
        p.re = qx;
        p.im = qy;
        cfx_mac(x, y, p, m[k]);
        m[3 + k].re = fx_split(fx_join(m[3 + k].re) - facc_get(x));
        m[3 + k].im = fx_split(fx_join(m[3 + k].im) - facc_get(y));
    }
    const long long d1 = fx_row_norm2(m + 3) - one;
    fx_scale_row(m + 3, fx_rsqrt1(d1));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        facc x = facc_zero(), y = facc_zero(), u = facc_zero(), v = facc_zero();
        cfx_mac(x, y, m[i], m[3 + j]);
        cfx_mac(u, v, m[j], m[3 + i]);
        m[6 + k].re = fx_split(facc_get(x) - facc_get(u));
        m[6 + k].im = fx_split(facc_get(v) - facc_get(y));
    }
    return fx_far(d0) || fx_far(d1);
}

#ifdef __CUDACC__
// ---- loads of FP64 and FP32 matrices ---------------------------------------------
// Matrices the fixed-point kernels do not take (callers' unvalidated fields): an
// entry above 1.03 in magnitude or not finite, or a row whose squared norm is
// off 1 by 5 % (tiny rows would lose relative precision).  Unit rows need not be
// orthogonal: a matrix that passes has a spectral norm of up to 1.78.  Kernels
// whose sums need more than that allows take fx_bad_gram (fx_load_unitary) as
// well: squared row norms within 2 % of 1 and row inner products of components
// below 1 %, which bounds the spectral norm by 1.024 (the Gram matrix less 1 has
// a norm below 0.02 + 2 sqrt(2) 0.01).
__device__ __forceinline__ unsigned fx_magnitude(double d) { return __double2hiint(d) & 0x7fffffff; }
__device__ __forceinline__ unsigned fx_magnitude(float f) {  // as the high word of the same double, roughly
    return ((__float_as_uint(f) & 0x7fffffff) >> 3) + 0x38000000u;
}
__device__ __forceinline__ fx fx_of(float f) {
    const float s = f * 0x1p28f;
    const int h = __float2int_rn(s);
    return fx_split(((long long)h << 32) + 2 * (long long)__float2int_rn((s - (float)h) * 0x1p31f));
}
constexpr unsigned kFxMagnitude = 0x3ff07ae1;  // 1.03
__device__ __forceinline__ bool fx_bad_rows(const cfx* m) {
    bool bad = false;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        float n2 = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float x = (float)m[3 * r + k].re.h, y = (float)m[3 * r + k].im.h;  // unit 2^-28
            n2 = fmaf(x, x, fmaf(y, y, n2));
        }
        bad = bad || !(fabsf(n2 * 0x1p-56f - 1.f) < 0.05f);
    }
    return bad;
}
__device__ __forceinline__ bool fx_bad_gram(const cfx* m) {
    bool bad = false;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int q = r; q < 3; ++q) {
            float re = 0.f, im = 0.f;  // conj(row r) . row q, unit 2^-56
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float ax = (float)m[3 * r + k].re.h, ay = (float)m[3 * r + k].im.h;
                const float bx = (float)m[3 * q + k].re.h, by = (float)m[3 * q + k].im.h;
                re = fmaf(ax, bx, fmaf(ay, by, re));
                im = fmaf(ax, by, fmaf(-ay, bx, im));
            }
            bad = bad || (q == r ? !(fabsf(re * 0x1p-56f - 1.f) < 0.02f)
                                 : !(fmaxf(fabsf(re), fabsf(im)) * 0x1p-56f < 0.01f));
        }
    return bad;
}
// entry (r, k) at src[r sr + k sc] to m; true: an entry or a row norm out of range
template <typename C>
__device__ __forceinline__ bool fx_load_matrix(const C* __restrict__ src, size_t sr, size_t sc, cfx* m) {
    unsigned big = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const C d = src[r * sr + k * sc];
            big = max(big, max(fx_magnitude(d.x), fx_magnitude(d.y)));
            m[3 * r + k].re = fx_of(d.x);
            m[3 * r + k].im = fx_of(d.y);
        }
    return big > kFxMagnitude || fx_bad_rows(m);
}
// the same; true: not near-unitary
__device__ __forceinline__ bool fx_load_unitary(const double2* __restrict__ src, size_t sr, size_t sc, cfx* m) {
    const bool bad = fx_load_matrix(src, sr, sc, m);
    return fx_bad_gram(m) || bad;
}
__device__ __forceinline__ bool fx_bad_matrix(const double2* src, size_t sr, size_t sc) {
    cfx m[9];
    return fx_load_unitary(src, sr, sc, m);
}
// X 2^-60 rounded to FP32 (ties away from zero)
__device__ __forceinline__ float fx_single(long long X) {
    const long long sg = X >> 63;
    const unsigned long long m = (unsigned long long)((X ^ sg) - sg);
    const int z = __clzll((long long)m);
    const unsigned t = (unsigned)((z > 0 ? m << ((z - 1) & 63) : m >> 1) >> 32);  // top bit 30
    // the bits below the upper word only matter for a tie, which then rounds up as well
    const unsigned q = ((t + (1u << 6)) >> 7) + ((unsigned)(129 - z) << 23);
    return __uint_as_float(X == 0 ? 0u : (q | ((unsigned)sg & 0x80000000u)));
}
__device__ __forceinline__ void fx_store(double2* p, cfx v) {
    *p = make_double2(fx_double(fx_join(v.re)), fx_double(fx_join(v.im)));
}
__device__ __forceinline__ void fx_store(float2* p, cfx v) {
    *p = make_float2(fx_single(fx_join(v.re)), fx_single(fx_join(v.im)));
}
__device__ __forceinline__ cfx fx_load(const int4* p) {
    const int4 v = *p;
    cfx r;
    r.re.h = v.x;
    r.re.l = v.y;
    r.im.h = v.z;
    r.im.l = v.w;
    return r;
}
__device__ __forceinline__ int4 fx_pack(cfx a) { return make_int4(a.re.h, a.re.l, a.im.h, a.im.l); }
#endif

}  // namespace mcg
