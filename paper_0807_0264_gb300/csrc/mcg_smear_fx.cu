// FP64 smearing in fixed-point arithmetic (mcg_fx.cuh): the step of
// mcg_smear.cu on fields held as 64-bit integers of unit 2^-60.
#include <cuda_runtime.h>

#include <cmath>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"

namespace mcg {

// One factor of a staple path: link direction (0: mu, 1: nu), displacement
// (dm along mu, dn along nu) of its site from x, daggered or not.
struct FxPathFactor {
    signed char dir, dm, dn, dag;
};
// The 8 staple shapes per nu != mu: two plaquette staples, then the six
// rectangle staples (1x2 up/down, 2x1 forward up/down, 2x1 backward up/down),
// each a path from x to x + mu.
__constant__ FxPathFactor c_fx_paths[8][5] = {
    {{1, 0, 0, 0}, {0, 0, 1, 0}, {1, 1, 0, 1}, {0, 0, 0, 0}, {0, 0, 0, 0}},
    {{1, 0, -1, 1}, {0, 0, -1, 0}, {1, 1, -1, 0}, {0, 0, 0, 0}, {0, 0, 0, 0}},
    {{1, 0, 0, 0}, {1, 0, 1, 0}, {0, 0, 2, 0}, {1, 1, 1, 1}, {1, 1, 0, 1}},
    {{1, 0, -1, 1}, {1, 0, -2, 1}, {0, 0, -2, 0}, {1, 1, -2, 0}, {1, 1, -1, 0}},
    {{1, 0, 0, 0}, {0, 0, 1, 0}, {0, 1, 1, 0}, {1, 2, 0, 1}, {0, 1, 0, 1}},
    {{1, 0, -1, 1}, {0, 0, -1, 0}, {0, 1, -1, 0}, {1, 2, -1, 0}, {0, 1, 0, 1}},
    {{0, -1, 0, 1}, {1, -1, 0, 0}, {0, -1, 1, 0}, {0, 0, 1, 0}, {1, 1, 0, 1}},
    {{0, -1, 0, 1}, {1, -1, -1, 1}, {0, -1, -1, 0}, {0, 0, -1, 0}, {1, 1, -1, 0}},
};

constexpr int kFxTerms = 28;  // series terms of exp(iQ) at most

struct FxSmear {
    fx wp, wr;           // rho times the plaquette weight; 8 rho times the rectangle weight
    fx third;            // 1/3
    fx term[kFxTerms];   // i^k 2^k / k! without the factor i of odd k (sign of k % 4 in {2, 3}: minus)
    int nterms;          // even
};

// factor f of a staple path of the link (mu, c): its matrix, daggered (a
// transposed read with the imaginary parts negated) where the path asks for it
__device__ __forceinline__ void fx_factor(const int4* __restrict__ U, const Geom& g, const int c[4], int mu, int nu,
                                          FxPathFactor f, cfx* m) {
    int q[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const int v = c[d] + (d == mu ? f.dm : 0) + (d == nu ? f.dn : 0);
        q[d] = v < 0 ? v + g.n[d] : (v >= g.n[d] ? v - g.n[d] : v);
    }
    const int p = (q[0] + q[1] + q[2] + q[3]) & 1;
    const int4* base = U + lidx(g, f.dir ? nu : mu, p, 0, eo_index(g, q));
    const size_t sr = (size_t)g.vh * (f.dag ? 1 : 3), sc = (size_t)g.vh * (f.dag ? 3 : 1);
    const int sg = f.dag ? -1 : 1;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cfx v = fx_load(base + i * sr + j * sc);
            v.im.h *= sg;
            v.im.l *= sg;
            m[3 * i + j] = v;
        }
}

__device__ __forceinline__ long long fx_abs2(cfx a) {
    facc s = facc_zero();
    fx_mac(s, a.re, a.re);
    fx_mac(s, a.im, a.im);
    return facc_get(s);
}

// exp(iQ) with Q = 2 x, x traceless Hermitian of spectral radius at most 0.67:
// diagonal d, upper triangle x01, x02, x12.  Powers of x reduce by
// Cayley-Hamilton, x^3 = c1 x + c0 with c1 = tr x^2 / 2, c0 = det x:
// x^k = a_k + b_k x + b_{k-1} x^2 with a_k = c0 b_{k-2} and
// b_{k+1} = c1 b_{k-1} + c0 b_{k-2}, so
// exp(iQ) = sum_k (2^k / k!) i^k x^k = f0 + f1 x + f2 x^2 needs one three-term
// recurrence of reals.  (No square root, division or angle, and no case near
// degenerate eigenvalues.)
__device__ __forceinline__ void fx_exp(const fx (&d)[3], cfx x01, cfx x02, cfx x12, const FxSmear& P, cfx* E) {
    const long long n01 = fx_abs2(x01), n02 = fx_abs2(x02), n12 = fx_abs2(x12);
    const long long s0 = fx_mul(d[0], d[0]), s1 = fx_mul(d[1], d[1]), s2 = fx_mul(d[2], d[2]);
    const long long c1 = ((s0 + s1 + s2) >> 1) + n01 + n02 + n12;
    // det: d0 d1 d2 + 2 Re(x01 x12 conj(x02)) - d0 |x12|^2 - d1 |x02|^2 - d2 |x01|^2
    facc u = facc_zero(), v = facc_zero();
    cfx_mac(u, v, x01, x12);
    const cfx x0112 = cfx_get(u, v);
    facc t = facc_zero();
    fx_mac(t, x0112.re, x02.re);
    fx_mac(t, x0112.im, x02.im);
    const long long re2 = 2 * facc_get(t);
    t = facc_zero();
    fx_mac(t, fx_split(fx_mul(d[0], d[1])), d[2]);
    fx_msc(t, d[0], fx_split(n12));
    fx_msc(t, d[1], fx_split(n02));
    fx_msc(t, d[2], fx_split(n01));
    const fx c0 = fx_split(facc_get(t) + re2), c1s = fx_split(c1);

    facc f1r = facc_zero(), f1i = facc_zero(), f2r = facc_zero(), f2i = facc_zero(), gr = facc_zero(),
         gi = facc_zero();
    fx b2 = {0, 0}, b1 = {1 << 28, 0}, b = {0, 0};  // b_{k-2}, b_{k-1}, b_k at k = 2
    fx_mac(f1i, P.term[1], b1);
#pragma unroll 1
    for (int k = 2; k < P.nterms; k += 2) {
        const fx te = P.term[k], to = P.term[k + 1];
        fx_mac(f1r, te, b);
        fx_mac(f2r, te, b1);
        fx_mac(gr, te, b2);
        facc s = facc_zero();
        fx_mac(s, c1s, b1);
        fx_mac(s, c0, b2);
        fx n = fx_split(facc_get(s));
        fx_mac(f1i, to, n);
        fx_mac(f2i, to, b);
        fx_mac(gi, to, b1);
        s = facc_zero();
        fx_mac(s, c1s, b);
        fx_mac(s, c0, b1);
        b2 = b;
        b1 = n;
        b = fx_split(facc_get(s));
    }
    const cfx f1 = cfx_get(f1r, f1i), f2 = cfx_get(f2r, f2i);
    cfx f0;
    f0.re = fx_split(fx_mul(fx_split(facc_get(gr)), c0) + (1LL << 60));
    f0.im = fx_split(fx_mul(fx_split(facc_get(gi)), c0));

    const long long y[3] = {s0 + n01 + n02, s1 + n01 + n12, s2 + n02 + n12};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const fx yi = fx_split(y[i]);
        facc r = facc_zero(), m = facc_zero();
        fx_mac(r, f1.re, d[i]);
        fx_mac(r, f2.re, yi);
        fx_mac(m, f1.im, d[i]);
        fx_mac(m, f2.im, yi);
        E[4 * i].re = fx_split(facc_get(r) + fx_join(f0.re));
        E[4 * i].im = fx_split(facc_get(m) + fx_join(f0.im));
    }
    // off-diagonal entries of x^2: y01 = x02 conj(x12) - d2 x01, y02 = x01 x12 - d1 x02,
    // y12 = conj(x01) x02 - d0 x12
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const cfx x = q == 0 ? x01 : (q == 1 ? x02 : x12);
        facc r = facc_zero(), m = facc_zero();
        if (q == 0)
            cfx_macc(r, m, x02, x12);
        else if (q == 1)
            cfx_mac(r, m, x01, x12);
        else
            cfx_macc(r, m, x02, x01);
        const fx dd = d[2 - q];
        fx_msc(r, dd, x.re);
        fx_msc(m, dd, x.im);
        const cfx yq = cfx_get(r, m);
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        facc p = facc_zero(), w = facc_zero();
        cfx_mac(p, w, f1, x);
        cfx_mac(p, w, f2, yq);
        E[3 * i + j] = cfx_get(p, w);
        p = facc_zero();
        w = facc_zero();
        cfx_macc(p, w, f1, x);
        cfx_macc(p, w, f2, yq);
        E[3 * j + i] = cfx_get(p, w);
    }
}

// One thread per link, old field in, new field out (fixed point, or FP64 after
// the last step).  The staples run over the table of paths with one rolled
// product body (a small loop body keeps the instruction fetch out of the way;
// a daggered factor is a transposed read; with a second body for it the
// stout step took 12 % longer).  Bounds: links have entries and row
// norms at most 1 (+1e-6), so has every path; the plaquette sum of six paths
// stays below 8, the sum of 18 rectangles is kept in units of 8; the caller
// guarantees |rho| (6 |cp| + 18 |cr|) <= 1, which bounds C's rows by 1 and Q's
// spectral radius by 4/3.
// Bound by the integer multiplier.  Measured on 20^3 x 40: 0.96 ms per stout
// step (the FP64 kernel: 4.88 ms, FP64 pipe 93 % busy); over-improved steps on
// 12 x 10 x 14 x 22: 0.63 ms (2.70 ms).  3 blocks of 128 per SM: 2 blocks take
// 12 %, 4 (spilling) 4 % longer.  Deviation from a 128-bit reference (4^4, ten
// stout steps): 7.5e-17 rms, the FP64 kernel's 2.2e-16.
template <bool RECT, bool OUT64>
__global__ void __launch_bounds__(128, 3) k_smear_step_fx(const int4* __restrict__ Uin, int4* __restrict__ Uout,
                                                          Geom g, int nfields, const __grid_constant__ FxSmear P) {
    const long long n = 8LL * g.vh * nfields;
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= n) return;
    const int f = (int)(id / (8LL * g.vh));
    int r = (int)(id - (long long)f * 8 * g.vh);
    const int mu = r / (2 * g.vh);
    r -= mu * 2 * g.vh;
    const int p = r / g.vh, s = r - p * g.vh;
    const int4* U = Uin + (size_t)f * link_elems(g);
    int c[4];
    eo_coords(g, p, s, c);

    long long C[18];
#pragma unroll
    for (int e = 0; e < 18; ++e) C[e] = 0;
    cfx a[9], b[9];
    // rectangles first, then (weighted) plaquettes: one sum in registers
#pragma unroll 1
    for (int k = RECT ? 7 : 1; k >= 0; --k) {
        const int nf = k < 2 ? 3 : 5;
        if (RECT && k == 1) {
#pragma unroll
            for (int e = 0; e < 18; ++e) C[e] = fx_mul(fx_split(C[e]), P.wr);
        }
#pragma unroll 1
        for (int nu = 0; nu < 4; ++nu) {
            if (nu == mu) continue;
            fx_factor(U, g, c, mu, nu, c_fx_paths[k][0], a);
#pragma unroll 1
            for (int j = 1; j < nf; ++j) {
                fx_factor(U, g, c, mu, nu, c_fx_paths[k][j], b);
                m3fx_mul_inplace<false>(a, b);
            }
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                if (!RECT) {
                    C[2 * e] += fx_join(a[e].re);
                    C[2 * e + 1] += fx_join(a[e].im);
                } else if (k < 2) {
                    C[2 * e] += fx_mul(a[e].re, P.wp);
                    C[2 * e + 1] += fx_mul(a[e].im, P.wp);
                } else {
                    C[2 * e] += fx_join(a[e].re) >> 3;
                    C[2 * e + 1] += fx_join(a[e].im) >> 3;
                }
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        a[e].re = fx_split(RECT ? C[2 * e] : fx_mul(fx_split(C[2 * e]), P.wp));
        a[e].im = fx_split(RECT ? C[2 * e + 1] : fx_mul(fx_split(C[2 * e + 1]), P.wp));
    }
    // Omega = C U^dag, x = Q / 2 = (i/4) (Omega^dag - Omega) less its trace
    const int4* ul = U + lidx(g, mu, p, 0, s);
#pragma unroll
    for (int e = 0; e < 9; ++e) b[e] = fx_load(ul + (size_t)e * g.vh);
    m3fx_mul_inplace<true>(a, b);
    const cfx* om = a;
    const long long o0 = fx_join(om[0].im), o1 = fx_join(om[4].im), o2 = fx_join(om[8].im);
    const long long mean = fx_mul(fx_split(o0 + o1 + o2), P.third);
    const long long h0 = (o0 - mean) >> 1, h1 = (o1 - mean) >> 1;
    const fx d[3] = {fx_split(h0), fx_split(h1), fx_split(-h0 - h1)};
    cfx x[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        x[q].re = fx_split((fx_join(om[3 * j + i].im) + fx_join(om[3 * i + j].im)) >> 2);
        x[q].im = fx_split((fx_join(om[3 * j + i].re) - fx_join(om[3 * i + j].re)) >> 2);
    }
    fx_exp(d, x[0], x[1], x[2], P, a);
    m3fx_mul_inplace<false>(a, b);
    int4* out = Uout + (size_t)f * link_elems(g) + lidx(g, mu, p, 0, s);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        if (OUT64) {
            reinterpret_cast<double2*>(out)[(size_t)e * g.vh] =
                make_double2(fx_double(fx_join(a[e].re)), fx_double(fx_join(a[e].im)));
        } else {
            out[(size_t)e * g.vh] = fx_pack(a[e]);
        }
    }
}

// n complex FP64 numbers of magnitude below 8 -> fixed point
__global__ void __launch_bounds__(256) k_to_fx(const double2* __restrict__ src, int4* __restrict__ dst, size_t n) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double2 v = src[k];
    cfx r;
    r.re = fx_of(v.x);
    r.im = fx_of(v.y);
    dst[k] = fx_pack(r);
}

bool smear_fx_applies(double rho, double eps) {
    const double cp = (5.0 - 2.0 * eps) / 3.0, cr = -(1.0 - eps) / 12.0;
    return std::fabs(rho) * (6.0 * std::fabs(cp) + 18.0 * std::fabs(cr)) <= 1.0;
}

static fx host_fx(double v) { return fx_split(std::llrint(std::ldexp(v, 60))); }

int run_smear_fx(const void* Uin, void* Uout, const Geom& g, int nfields, double rho, double eps, int n,
                 cudaStream_t st) {
    const size_t elems = link_elems(g) * (size_t)nfields;
    int rc = 0;
    void* tmp = scratch_device("smear.tmp", 16 * elems, &rc);
    if (rc) return rc;
    const double cp = (5.0 - 2.0 * eps) / 3.0, cr = -(1.0 - eps) / 12.0;
    const bool rect = cr != 0.0;
    FxSmear P;
    P.wp = host_fx(rho * cp);
    P.wr = host_fx(8.0 * rho * cr);
    P.third = fx_split(((1LL << 60) + 1) / 3);
    // 2^k / k! with 40 guard bits, rounded to 2^-60; terms until the bound
    // r^k / k! on the rest is below 2^-62, r = 4/3 of the staple weight
    const double rad = 4.0 / 3.0 * std::fabs(rho) * (6.0 * std::fabs(cp) + 18.0 * std::fabs(cr));
    unsigned __int128 t = (unsigned __int128)1 << 100;
    double rest = 1.0;
    P.nterms = 0;
    for (int k = 0; k < kFxTerms; ++k) {
        if (k > 0) {
            t = t * 2 / k;
            rest *= rad / k;
        }
        const long long X = (long long)((t + ((unsigned __int128)1 << 39)) >> 40);
        P.term[k] = fx_split((k % 4) >= 2 ? -X : X);
        if (P.nterms == 0 && k >= 8 && k % 2 == 0 && rest < 0x1p-62) P.nterms = k;
    }
    if (P.nterms == 0) P.nterms = kFxTerms;
    // step k's source: tmp or Uout in turn, so that the last step reads tmp
    auto buf = [&](int k) { return (n - 1 - k) % 2 == 0 ? tmp : Uout; };
    const unsigned cb = (unsigned)((elems + 255) / 256);
    k_to_fx<<<cb, 256, 0, st>>>((const double2*)Uin, (int4*)buf(0), elems);
    const unsigned nb = (unsigned)((8LL * g.vh * nfields + 127) / 128);
    for (int k = 0; k < n; ++k) {
        const int4* src = (const int4*)buf(k);
        const bool last = k + 1 == n;
        int4* dst = (int4*)(last ? Uout : buf(k + 1));
        if (rect) {
            if (last)
                k_smear_step_fx<true, true><<<nb, 128, 0, st>>>(src, dst, g, nfields, P);
            else
                k_smear_step_fx<true, false><<<nb, 128, 0, st>>>(src, dst, g, nfields, P);
        } else {
            if (last)
                k_smear_step_fx<false, true><<<nb, 128, 0, st>>>(src, dst, g, nfields, P);
            else
                k_smear_step_fx<false, false><<<nb, 128, 0, st>>>(src, dst, g, nfields, P);
        }
    }
    MCG_CK(cudaGetLastError());
    note_launches(n + 1);
    return 0;
}

// index-check counter of this unit (MCG_CHECK builds)
MCG_BOUND_READER(bound_hits_smear_fx)

}  // namespace mcg
