// Device code of the smearing steps in fixed point (forward: mcg_smear_fx.cu,
// reverse mode: mcg_smear_bwd_fx.cu): staple paths, the staple sum of a link and
// the generator Q of its step.
#pragma once

#include <cuda_runtime.h>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"

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

// The caller guarantees |rho| (6 |cp| + 18 |cr|) <= 1 (smear_fx_applies), which
// bounds the rows of the weighted staple sum by 1 and the spectral radius of Q by
// 4/3.
struct FxSmear {
    fx wp, wr;           // rho times the plaquette weight; 8 times rho times the rectangle weight
    fx gp, gr64;         // for gradients: wp and 8 wr times 2^gs, the weights of all staples
    int gs;              // together then between 1/2 and 1 (small rho: no loss of digits)
    fx third;            // 1/3
    fx term[kFxTerms];   // i^k 2^k / k! without the factor i of odd k (sign of k % 4 in {2, 3}: minus)
    int nterms;          // even
};

// The nine entries at base (stride vh); dag: of the adjoint, a transposed read
// with the imaginary parts negated.  Addresses and signs by additions: products
// for them go to the multiplier, which bounds the callers (3.5 % of a smearing
// step).
__device__ __forceinline__ void fx_load_entries(const int4* __restrict__ base, size_t vh, bool dag, cfx* m) {
    const size_t sr = vh * (dag ? 16 : 48), sc = vh * (dag ? 48 : 16);
    const int sg = dag ? -1 : 0;
    const char* row = reinterpret_cast<const char*>(base);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const char* q = row;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cfx v = fx_load(reinterpret_cast<const int4*>(q));
            v.im.h = (v.im.h ^ sg) - sg;
            v.im.l = (v.im.l ^ sg) - sg;
            m[3 * i + j] = v;
            q += sc;
        }
        row += sr;
    }
}

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
    fx_load_entries(U + lidx(g, f.dir ? nu : mu, p, 0, eo_index(g, q)), (size_t)g.vh, f.dag, m);
}

__device__ __forceinline__ long long fx_abs2(cfx a) {
    facc s = facc_zero();
    fx_mac(s, a.re, a.re);
    fx_mac(s, a.im, a.im);
    return facc_get(s);
}

// Sum over the staples of the link (mu, c), weighted by rho and the staple
// weights, to C (rows bounded by 1, see FxSmear).  The staples run over the
// table of paths with one rolled product body (a small loop body keeps the
// instruction fetch out of the way; a daggered factor is a transposed read; with
// a second body for it the stout step took 12 % longer).  Rectangles first, then
// (weighted) plaquettes: one sum in registers.  Links have entries and row norms
// at most 1 (spectral norms of 1.024 for unvalidated ones, fx_bad_gram, and 1.13
// for a path of five), so has every path; the
// plaquette sum of six paths stays below 8, the sum of 18 rectangles is kept in
// units of 8.
template <bool RECT>
__device__ __forceinline__ void fx_staple_sum(const int4* __restrict__ U, const Geom& g, const int c[4], int mu,
                                              const FxSmear& P, cfx* a, cfx* b) {
    long long C[18];
#pragma unroll
    for (int e = 0; e < 18; ++e) C[e] = 0;
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
}

// x = Q / 2 = (i/4) (Omega^dag - Omega) less its trace, for Omega = C U^dag:
// diagonal d, upper triangle x (01, 02, 12)
__device__ __forceinline__ void fx_generator(const cfx* om, fx third, fx (&d)[3], cfx (&x)[3]) {
    const long long o0 = fx_join(om[0].im), o1 = fx_join(om[4].im), o2 = fx_join(om[8].im);
    const long long mean = fx_mul(fx_split(o0 + o1 + o2), third);
    const long long h0 = (o0 - mean) >> 1, h1 = (o1 - mean) >> 1;
    d[0] = fx_split(h0);
    d[1] = fx_split(h1);
    d[2] = fx_split(-h0 - h1);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        x[q].re = fx_split((fx_join(om[3 * j + i].im) + fx_join(om[3 * i + j].im)) >> 2);
        x[q].im = fx_split((fx_join(om[3 * j + i].re) - fx_join(om[3 * i + j].re)) >> 2);
    }
}

// invariants of x: c1 = tr x^2 / 2, c0 = det x, and x^2 (diagonal y; its upper
// triangle by fx_square_upper)
__device__ __forceinline__ void fx_invariants(const fx (&d)[3], const cfx (&x)[3], fx& c0, fx& c1, fx (&y)[3]) {
    const long long n01 = fx_abs2(x[0]), n02 = fx_abs2(x[1]), n12 = fx_abs2(x[2]);
    const long long s0 = fx_mul(d[0], d[0]), s1 = fx_mul(d[1], d[1]), s2 = fx_mul(d[2], d[2]);
    c1 = fx_split(((s0 + s1 + s2) >> 1) + n01 + n02 + n12);
    // det: d0 d1 d2 + 2 Re(x01 x12 conj(x02)) - d0 |x12|^2 - d1 |x02|^2 - d2 |x01|^2
    facc u = facc_zero(), v = facc_zero();
    cfx_mac(u, v, x[0], x[2]);
    const cfx x0112 = cfx_get(u, v);
    facc t = facc_zero();
    fx_mac(t, x0112.re, x[1].re);
    fx_mac(t, x0112.im, x[1].im);
    const long long re2 = 2 * facc_get(t);
    t = facc_zero();
    fx_mac(t, fx_split(fx_mul(d[0], d[1])), d[2]);
    fx_msc(t, d[0], fx_split(n12));
    fx_msc(t, d[1], fx_split(n02));
    fx_msc(t, d[2], fx_split(n01));
    c0 = fx_split(facc_get(t) + re2);
    y[0] = fx_split(s0 + n01 + n02);
    y[1] = fx_split(s1 + n01 + n12);
    y[2] = fx_split(s2 + n02 + n12);
}
// entry q (01, 02, 12) of x^2: x02 conj(x12) - d2 x01, x01 x12 - d1 x02,
// conj(x01) x02 - d0 x12
template <int Q>
__device__ __forceinline__ cfx fx_square_upper(const fx (&d)[3], const cfx (&x)[3]) {
    facc r = facc_zero(), m = facc_zero();
    if (Q == 0)
        cfx_macc(r, m, x[1], x[2]);
    else if (Q == 1)
        cfx_mac(r, m, x[0], x[2]);
    else
        cfx_macc(r, m, x[1], x[0]);
    fx_msc(r, d[2 - Q], x[Q].re);
    fx_msc(m, d[2 - Q], x[Q].im);
    return cfx_get(r, m);
}

// E = f0 + f1 x + f2 x^2
__device__ __forceinline__ void fx_exp_matrix(const fx (&d)[3], const cfx (&x)[3], const fx (&y)[3], cfx f0, cfx f1,
                                              cfx f2, cfx* E) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        facc r = facc_zero(), m = facc_zero();
        fx_mac(r, f1.re, d[i]);
        fx_mac(r, f2.re, y[i]);
        fx_mac(m, f1.im, d[i]);
        fx_mac(m, f2.im, y[i]);
        E[4 * i].re = fx_split(facc_get(r) + fx_join(f0.re));
        E[4 * i].im = fx_split(facc_get(m) + fx_join(f0.im));
    }
    const cfx yu[3] = {fx_square_upper<0>(d, x), fx_square_upper<1>(d, x), fx_square_upper<2>(d, x)};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        facc p = facc_zero(), w = facc_zero();
        cfx_mac(p, w, f1, x[q]);
        cfx_mac(p, w, f2, yu[q]);
        E[3 * i + j] = cfx_get(p, w);
        p = facc_zero();
        w = facc_zero();
        cfx_macc(p, w, f1, x[q]);
        cfx_macc(p, w, f2, yu[q]);
        E[3 * j + i] = cfx_get(p, w);
    }
}

// FxSmear for one pair of parameters (mcg_smear_fx.cu); slack: factor on the
// staple weight in the truncation bound
FxSmear fx_smear_params(double rho, double eps, double slack);
// n complex FP64 numbers of magnitude below 8 -> fixed point
void launch_to_fx(const void* src, void* dst, size_t n, cudaStream_t st);

}  // namespace mcg
