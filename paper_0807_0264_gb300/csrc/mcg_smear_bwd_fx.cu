// Reverse mode of one FP64 smearing step in fixed-point arithmetic (mcg_fx.cuh),
// without atomics: pass 1 turns each link's output gradient into its adjoint
// matrix, pass 2 gathers, for each link, its part in every staple that holds it.
//
// Gradients have no bound of their own, so each matrix carries a power of two:
// pass 1 scales a link's gradient to components below 1/2 (exponent e), pass 2
// brings the matrices that reach a link through its staples to the largest
// exponent among them (block floating point: an error of 2^-57 of the largest,
// times the staples' weight, which a power of two keeps between 1/2 and 1 until the
// end).  The link's own part keeps its own exponent, so that it loses nothing beside
// large neighbours, at rho = 0 not even a digit.
#include <cuda_runtime.h>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"
#include "mcg_smear_fx.cuh"

namespace mcg {

namespace {

inline unsigned blocks(long long n, int nt) { return (unsigned)((n + nt - 1) / nt); }

// d 2^-e as an integer of unit 2^-60, |d| 2^-e < 1/2, e = (largest exponent
// field) - 1021
__device__ __forceinline__ fx fx_of_scaled(double d, int e) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
    const int field = (int)((bits >> 52) & 0x7ff), r = 1025 + e - field;
    const unsigned long long m = ((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
    const unsigned long long v = r > 63 || field == 0 ? 0ULL : m >> (r & 63);
    const long long sg = (long long)bits >> 63;
    return fx_split(((long long)v ^ sg) - sg);
}
// X 2^(e - 60)
__device__ __forceinline__ double fx_double_scaled(long long X, int e) {
    const long long sg = X >> 63;
    unsigned long long m = (unsigned long long)((X ^ sg) - sg);
    const int z = __clzll((long long)m);
    m = z > 0 ? m << ((z - 1) & 63) : m >> 1;
    const int field = 1025 - z + e;
    const unsigned long long q = ((m + (1ULL << 9)) >> 10) + ((unsigned long long)(unsigned)max(field, 0) << 52);
    const unsigned long long s = (unsigned long long)sg & 0x8000000000000000ULL;
    const unsigned long long inf = 0x7ff0000000000000ULL;
    return __longlong_as_double((long long)(X == 0 || field < 0 ? 0ULL : (field > 2045 ? s | inf : s | q)));
}

// links to fixed point, one thread per matrix; bad counts those that are not
// near-unitary
__global__ void __launch_bounds__(128) k_links_to_fx(const double2* __restrict__ src, int4* __restrict__ dst, size_t vh,
                                                     long long nmat, unsigned* __restrict__ bad) {
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= nmat) return;
    const size_t o = (size_t)(id / (long long)vh) * 9 * vh + (size_t)(id % (long long)vh);
    cfx m[9];
    if (fx_load_unitary(src + o, 3 * vh, vh, m)) atomicAdd(bad, 1u);
#pragma unroll
    for (int e = 0; e < 9; ++e) dst[o + e * vh] = fx_pack(m[e]);
}

__device__ __forceinline__ cfx cfx_prod(cfx a, cfx b) {
    facc x = facc_zero(), y = facc_zero();
    cfx_mac(x, y, a, b);
    return cfx_get(x, y);
}
__device__ __forceinline__ cfx cfx_prod2(cfx a, cfx b, cfx c, cfx d) {  // a b + c d
    facc x = facc_zero(), y = facc_zero();
    cfx_mac(x, y, a, b);
    cfx_mac(x, y, c, d);
    return cfx_get(x, y);
}
__device__ __forceinline__ cfx cfx_scale(fx s, cfx a) {
    cfx r;
    r.re = fx_split(fx_mul(s, a.re));
    r.im = fx_split(fx_mul(s, a.im));
    return r;
}
__device__ __forceinline__ cfx cfx_add(cfx a, cfx b) {
    cfx r;
    r.re = fx_split(fx_join(a.re) + fx_join(b.re));
    r.im = fx_split(fx_join(a.im) + fx_join(b.im));
    return r;
}
__device__ __forceinline__ cfx cfx_conj(cfx a) {
    a.im = fx_neg(a.im);
    return a;
}
// tr(h m) for the Hermitian h (diagonal d, upper triangle u)
__device__ __forceinline__ cfx trace_hermitian(const fx (&d)[3], const cfx (&u)[3], const cfx* m) {
    facc x = facc_zero(), y = facc_zero();
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        fx_mac(x, d[i], m[4 * i].re);
        fx_mac(y, d[i], m[4 * i].im);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        cfx_mac(x, y, u[q], m[3 * j + i]);
        cfx_macc(x, y, m[3 * i + j], u[q]);
    }
    return cfx_get(x, y);
}

// Pass 1, one thread per link.  With E = exp(iQ), C the weighted staple sum and
// G the output gradient: K, the traceless anti-Hermitian part of the Frechet
// derivative of exp at iQ in the direction U G^dag; out go E^dag G + K C (the
// link's own part, to D) and U^dag K (to Y), both in units of 2^(e - 60).
//
// The derivative comes from the closed form exp(iQ) = f0 + f1 x + f2 x^2 (x =
// Q / 2, f_j functions of c0 = det x and c1 = tr x^2 / 2): along dx = -(i/2) of
// the direction's traceless part,
//   L = f1 dx + f2 (dx x + x dx) + df1 x + df2 x^2 + df0, df_j = (d_0 f_j) dc0 + (d_1 f_j) dc1,
//   dc1 = tr(x dx), dc0 = tr(x^2 dx),
// and exp(iQ) times a third of its trace.  The f_j are sums over b_k (see
// fx_exp), their derivatives over d_k = d b_k / d c1, since d b_{k+1} / d c0 =
// d_k; d_{k+1} = b_{k-1} + c1 d_{k-1} + c0 d_{k-2}.  Seven products beside the
// staples, where the Taylor series of the block matrix took 72.
// The barriers hold no data: they keep the block's warps in step through ~100 KB
// of straight-line code, so that they share its instruction fetches (16^4: 424
// -> 363 us; 3 blocks per SM, spilling: 385).
template <bool RECT>
__global__ void __launch_bounds__(128, 2)
    k_smear_adjoint_fx(const int4* __restrict__ Uall, const double2* __restrict__ Gout, int4* __restrict__ Yall,
                       int4* __restrict__ Dall, int* __restrict__ exps, Geom g, int nfields,
                       const __grid_constant__ FxSmear P, unsigned* __restrict__ bad) {
    __shared__ int4 sC[9 * 128], sE[9 * 128];
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= 8LL * g.vh * nfields) return;
    const int f = (int)(id / (8LL * g.vh));
    int r = (int)(id - (long long)f * 8 * g.vh);
    const int mu = r / (2 * g.vh);
    r -= mu * 2 * g.vh;
    const int p = r / g.vh, s = r - p * g.vh;
    const size_t vh = (size_t)g.vh;
    const int4* U = Uall + (size_t)f * link_elems(g);
    const size_t o = (size_t)f * link_elems(g) + lidx(g, mu, p, 0, s);
    int c[4];
    eo_coords(g, p, s, c);

    // the gradient's exponent
    unsigned top = 0;
#pragma unroll 1
    for (int e = 0; e < 9; ++e) {
        const double2 v = Gout[o + e * vh];
        top = max(top, max(fx_magnitude(v.x), fx_magnitude(v.y)));
    }
    const int ef = (int)(top >> 20), e2 = ef - 1021;
    if (ef == 0x7ff) atomicAdd(bad, 1u);  // infinite or NaN: the FP64 kernel propagates it
    exps[id] = e2;

    cfx a[9], b[9];
    fx_staple_sum<RECT>(U, g, c, mu, P, a, b);
#pragma unroll
    for (int e = 0; e < 9; ++e) sC[e * 128 + threadIdx.x] = fx_pack(a[e]);
#pragma unroll
    for (int e = 0; e < 9; ++e) b[e] = fx_load(Uall + o + e * vh);
    m3fx_mul_inplace<true>(a, b);
    fx d[3], y[3], c0, c1;
    cfx x[3];
    __syncthreads();
    fx_generator(a, P.third, d, x);
    fx_invariants(d, x, c0, c1, y);

    // f_j and their derivatives
    cfx f0, f1, f2, df0[2], df1[2], df2[2];  // [0]: along c0, [1]: along c1
    {
        facc Br[3], Bi[3], Dr[4], Di[4];  // sums of b_{k-j} and d_{k-j} over even and odd k
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j < 3) Br[j] = Bi[j] = facc_zero();
            Dr[j] = Di[j] = facc_zero();
        }
        const fx zero = {0, 0}, one = {1 << 28, 0};
        fx bq[3] = {zero, one, zero}, dq[4] = {zero, zero, zero, zero};  // [j]: index k - j, k = 2
        fx_mac(Bi[0], P.term[1], one);
#pragma unroll 1
        for (int k = 2; k < P.nterms; k += 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const fx t = P.term[k + h];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j < 3) fx_mac(h ? Bi[j] : Br[j], t, bq[j]);
                    fx_mac(h ? Di[j] : Dr[j], t, dq[j]);
                }
                facc nb = facc_zero(), nd = facc_zero();
                fx_mac(nb, c1, bq[1]);
                fx_mac(nb, c0, bq[2]);
                fx_mac(nd, c1, dq[1]);
                fx_mac(nd, c0, dq[2]);
                const long long ndv = facc_get(nd) + fx_join(bq[1]);
                bq[2] = bq[1];
                bq[1] = bq[0];
                bq[0] = fx_split(facc_get(nb));
                dq[3] = dq[2];
                dq[2] = dq[1];
                dq[1] = dq[0];
                dq[0] = fx_split(ndv);
            }
        }
        f1 = cfx_get(Br[0], Bi[0]);
        f2 = cfx_get(Br[1], Bi[1]);
        const cfx gg = cfx_get(Br[2], Bi[2]);
        f0 = cfx_scale(c0, gg);
        f0.re = fx_split(fx_join(f0.re) + (1LL << 60));
        const cfx d0 = cfx_get(Dr[0], Di[0]), d1 = cfx_get(Dr[1], Di[1]), d2 = cfx_get(Dr[2], Di[2]),
                  d3 = cfx_get(Dr[3], Di[3]);
        df1[1] = d0;
        df1[0] = df2[1] = d1;
        df2[0] = d2;
        df0[1] = cfx_scale(c0, d2);
        df0[0] = cfx_add(gg, cfx_scale(c0, d3));
    }
    __syncthreads();
    fx_exp_matrix(d, x, y, f0, f1, f2, a);
#pragma unroll
    for (int e = 0; e < 9; ++e) sE[e * 128 + threadIdx.x] = fx_pack(a[e]);

    __syncthreads();
    // direction U G^dag: its traceless part as dx (in a), a third of its trace
    cfx tr3;
    {
        cfx gm[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const double2 v = Gout[o + e * vh];
            gm[e].re = fx_of_scaled(v.x, e2);
            gm[e].im = fx_of_scaled(v.y, e2);
            a[e] = b[e];
        }
        m3fx_mul_inplace<true>(a, gm);
    }
    tr3.re = fx_split(fx_mul(fx_split(fx_join(a[0].re) + fx_join(a[4].re) + fx_join(a[8].re)), P.third));
    tr3.im = fx_split(fx_mul(fx_split(fx_join(a[0].im) + fx_join(a[4].im) + fx_join(a[8].im)), P.third));
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const long long re = fx_join(a[e].re) - (e % 4 == 0 ? fx_join(tr3.re) : 0);
        const long long im = fx_join(a[e].im) - (e % 4 == 0 ? fx_join(tr3.im) : 0);
        a[e].re = fx_split(im >> 1);
        a[e].im = fx_split(-re >> 1);
    }
    __syncthreads();
    const cfx yu[3] = {fx_square_upper<0>(d, x), fx_square_upper<1>(d, x), fx_square_upper<2>(d, x)};
    const cfx dc1 = trace_hermitian(d, x, a), dc0 = trace_hermitian(y, yu, a);
    const cfx e0 = cfx_prod2(df0[0], dc0, df0[1], dc1), e1 = cfx_prod2(df1[0], dc0, df1[1], dc1),
              e2c = cfx_prod2(df2[0], dc0, df2[1], dc1);
    cfx n[9];
    {
        cfx xm[9];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            xm[4 * i].re = d[i];
            xm[4 * i].im.h = xm[4 * i].im.l = 0;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
            xm[3 * i + j] = x[q];
            xm[3 * j + i] = cfx_conj(x[q]);
        }
#pragma unroll
        for (int e = 0; e < 9; ++e) n[e] = a[e];
        m3fx_mul_inplace<false>(n, xm);
        m3fx_mul_inplace<false>(xm, a);
#pragma unroll
        for (int e = 0; e < 9; ++e) n[e] = cfx_add(n[e], xm[e]);
    }
    __syncthreads();
    // L, in a
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int e = 3 * i + j;
            cfx v = cfx_add(cfx_prod2(f1, a[e], tr3, fx_load(&sE[e * 128 + threadIdx.x])), cfx_prod(f2, n[e]));
            if (i == j) {
                v = cfx_add(v, e0);
                v = cfx_add(v, cfx_scale(d[i], e1));
                v = cfx_add(v, cfx_scale(y[i], e2c));
            } else {
                const int q = i + j - 1;
                v = cfx_add(v, i < j ? cfx_prod2(e1, x[q], e2c, yu[q])
                                     : cfx_prod2(e1, cfx_conj(x[q]), e2c, cfx_conj(yu[q])));
            }
            a[e] = v;
        }
    __syncthreads();
    // K = (L - L^dag) / 2 less its trace, in n
    const long long l0 = fx_join(a[0].im), l1 = fx_join(a[4].im), l2 = fx_join(a[8].im);
    const long long mean = fx_mul(fx_split(l0 + l1 + l2), P.third);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const long long re = (fx_join(a[3 * i + j].re) - fx_join(a[3 * j + i].re)) >> 1;
            long long im = (fx_join(a[3 * i + j].im) + fx_join(a[3 * j + i].im)) >> 1;
            if (i == j) im -= mean;
            n[3 * i + j].re = fx_split(re);
            n[3 * i + j].im = fx_split(im);
        }
    __syncthreads();
    // Y = U^dag K
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) a[3 * i + j] = cfx_conj(fx_load(Uall + o + (3 * j + i) * vh));
    m3fx_mul_inplace<false>(a, n);
#pragma unroll
    for (int e = 0; e < 9; ++e) Yall[o + e * vh] = fx_pack(a[e]);
    __syncthreads();
    // D = K C + E^dag G
#pragma unroll
    for (int e = 0; e < 9; ++e) b[e] = fx_load(&sC[e * 128 + threadIdx.x]);
    m3fx_mul_inplace<false>(n, b);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            a[3 * i + j] = cfx_conj(fx_load(&sE[(3 * j + i) * 128 + threadIdx.x]));
            const double2 v = Gout[o + (3 * i + j) * vh];
            b[3 * i + j].re = fx_of_scaled(v.x, e2);
            b[3 * i + j].im = fx_of_scaled(v.y, e2);
        }
    m3fx_mul_inplace<false>(a, b);
#pragma unroll
    for (int e = 0; e < 9; ++e) Dall[o + e * vh] = fx_pack(cfx_add(a[e], n[e]));
}

// site x + a mu + b nu, periodic; the link (dir, x) as an index of the field
__device__ __forceinline__ size_t link_at(const Geom& g, const int c[4], int dir, int mu, int a, int nu, int b) {
    int q[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        int v = c[d] + (d == mu ? a : 0) + (d == nu ? b : 0);
        while (v < 0) v += g.n[d];  // at most three steps on an extent of 2
        while (v >= g.n[d]) v -= g.n[d];
        q[d] = v;
    }
    const int p = (q[0] + q[1] + q[2] + q[3]) & 1;
    return lidx(g, dir, p, 0, eo_index(g, q));
}

// Pass 2, one thread per link (lam, z): the link is factor j of shape k of the
// staples of the links (mu, x) with mu = lam or sig, x = z minus the factor's
// displacement; its gradient takes Z = F_{j+1} ... F_{n-1} Y F_0 ... F_{j-1} (its
// adjoint where the factor is not daggered), times the staple's weight.  One
// rolled product body over the table of paths, as in the staple sum.  Matrices Y
// are shifted to the largest exponent of all that the link meets.  Their entries
// are at most 2.5 there, so the 18 plaquette terms are summed 3 bits lower and
// weighted at the end; with rectangles (90 more terms) each term is weighted
// before it is added, 1 bit lower (18 |wr| + 6 |wp| <= 1: the sums stay below 8).
// In place: D's entries are replaced by the FP64 gradient of the same link.
// Bound by the integer multiplier (83 % of its cycles; 16^4: 632 us).  Both
// passes take 1.0 ms per stout step at 16^4, the FP64 kernel with atomics 6.9 ms
// (33 ms at 20^3 x 40); the gradient's deviation from a 128-bit one is 0.9e-16 of
// its rms (1.0e-16 before).
template <bool RECT>
__global__ void __launch_bounds__(128, 3)
    k_smear_gather_fx(const int4* __restrict__ Uall, const int4* __restrict__ Yall, const int* __restrict__ exps,
                      int4* Gall, Geom g, int nfields, const __grid_constant__ FxSmear P,
                      const unsigned* __restrict__ bad) {
    if (*bad) return;  // the FP64 kernel redoes the step
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= 8LL * g.vh * nfields) return;
    const int f = (int)(id / (8LL * g.vh));
    int r = (int)(id - (long long)f * 8 * g.vh);
    const int lam = r / (2 * g.vh);
    r -= lam * 2 * g.vh;
    const int p = r / g.vh, s = r - p * g.vh;
    const size_t vh = (size_t)g.vh, foff = (size_t)f * link_elems(g);
    const int4* U = Uall + foff;
    const int4* Y = Yall + foff;
    const int* ex = exps + (size_t)f * 8 * vh;
    int c[4];
    eo_coords(g, p, s, c);

    // exponent of a link from its entry-0 index ((mu 2 + p) 9 vh + s)
    auto exponent = [&](size_t l) { return ex[(l / (9 * vh)) * vh + l % (9 * vh)]; };
    const int e_own = exps[id];
    int em = e_own;
#pragma unroll 1
    for (int k = RECT ? 7 : 1; k >= 0; --k)
#pragma unroll 1
        for (int sig = 0; sig < 4; ++sig) {
            if (sig == lam) continue;
#pragma unroll 1
            for (int j = 0; j < (k < 2 ? 3 : 5); ++j) {
                const FxPathFactor fj = c_fx_paths[k][j];
                const int mu = fj.dir ? sig : lam, nu = fj.dir ? lam : sig;
                em = max(em, exponent(link_at(g, c, mu, mu, -fj.dm, nu, -fj.dn)));
            }
        }

    long long S[18];
#pragma unroll
    for (int e = 0; e < 18; ++e) S[e] = 0;
    cfx a[9], b[9];
#pragma unroll 1
    for (int k = RECT ? 7 : 1; k >= 0; --k) {
        const int nf = k < 2 ? 3 : 5;
#pragma unroll 1
        for (int sig = 0; sig < 4; ++sig) {
            if (sig == lam) continue;
#pragma unroll 1
            for (int j = 0; j < nf; ++j) {
                const FxPathFactor fj = c_fx_paths[k][j];
                const int mu = fj.dir ? sig : lam, nu = fj.dir ? lam : sig;
#pragma unroll 1
                for (int t = 0; t < nf; ++t) {
                    const int m = j + 1 + t;
                    if (m == nf) {
                        const size_t l = link_at(g, c, mu, mu, -fj.dm, nu, -fj.dn);
                        const int sh = min(em - exponent(l) + (RECT ? 0 : 3), 63);
#pragma unroll
                        for (int e = 0; e < 9; ++e) {
                            const cfx v = fx_load(Y + l + e * vh);
                            b[e].re = fx_split(fx_join(v.re) >> sh);
                            b[e].im = fx_split(fx_join(v.im) >> sh);
                        }
                    } else {
                        const FxPathFactor ft = c_fx_paths[k][m < nf ? m : m - nf - 1];
                        const int4* q =
                            U + link_at(g, c, ft.dir ? nu : mu, mu, ft.dm - fj.dm, nu, ft.dn - fj.dn);
                        fx_load_entries(q, vh, ft.dag, b);
                    }
                    if (t == 0) {
#pragma unroll
                        for (int e = 0; e < 9; ++e) a[e] = b[e];
                    } else {
                        m3fx_mul_inplace<false>(a, b);
                    }
                }
                const bool dag = fj.dag;
                const fx w = k < 2 ? P.gp : P.gr64;
                const int ws = k < 2 ? 1 : 7, half = 1 << (ws - 1);
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int h = 0; h < 3; ++h) {
                        const int e = 3 * i + h, te = 3 * h + i;
                        long long re = fx_join(a[e].re), im = fx_join(a[e].im);
                        if (RECT) {
                            re = (fx_mul(fx_split(re), w) + half) >> ws;  // rounded: 108 floors add up
                            im = (fx_mul(fx_split(im), w) + half) >> ws;
                        }
                        S[2 * e] += dag ? re : 0;
                        S[2 * e + 1] += dag ? im : 0;
                        S[2 * te] += dag ? 0 : re;
                        S[2 * te + 1] -= dag ? 0 : im;
                    }
            }
        }
    }
    int4* out = Gall + foff + lidx(g, lam, p, 0, s);
    constexpr int up = RECT ? 1 : 3;
    if (!RECT) {
#pragma unroll
        for (int e = 0; e < 18; ++e) S[e] = fx_mul(fx_split(S[e]), P.gp);
    }
    // the link's own part in units of 2^(e_own - 60), the staples' in 2^(em + up - gs
    // - 60): one integer sum in units of 2^(em + up - 60) where that costs the own
    // part no digit that FP64 holds, else (a link whose gradient is far below its
    // neighbours') each to FP64 first
    const int sh = em - e_own + up, gs = min(P.gs, 63);
    if (sh <= 6) {
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const cfx v = fx_load(out + e * vh);
            const long long re = (fx_join(v.re) >> sh) + (S[2 * e] >> gs);
            const long long im = (fx_join(v.im) >> sh) + (S[2 * e + 1] >> gs);
            reinterpret_cast<double2*>(out)[e * vh] =
                make_double2(fx_double_scaled(re, em + up), fx_double_scaled(im, em + up));
        }
    } else {
#pragma unroll 1
        for (int e = 0; e < 9; ++e) {
            const cfx v = fx_load(out + e * vh);
            long long re = S[0], im = S[1];
#pragma unroll
            for (int k = 1; k < 9; ++k) {
                re = e == k ? S[2 * k] : re;
                im = e == k ? S[2 * k + 1] : im;
            }
            reinterpret_cast<double2*>(out)[e * vh] =
                make_double2(fx_double_scaled(fx_join(v.re), e_own) + fx_double_scaled(re, em + up - P.gs),
                             fx_double_scaled(fx_join(v.im), e_own) + fx_double_scaled(im, em + up - P.gs));
        }
    }
}

}  // namespace

int run_smear_backward_fx(const void* U, const double* Gout, double* Gin, const Geom& g, int nfields, double rho,
                          double eps, unsigned** bad_out, cudaStream_t st) {
    const size_t elems = link_elems(g) * (size_t)nfields;
    const long long nlinks = 8LL * g.vh * nfields;
    int4* Ufx = (int4*)scratch_device_optional("bwd.U", 16 * elems);
    int4* Y = (int4*)scratch_device_optional("bwd.Y", 16 * elems);
    int* ex = (int*)scratch_device_optional("bwd.exp", sizeof(int) * nlinks);
    unsigned* bad = (unsigned*)scratch_device_optional("bwd.bad", sizeof(unsigned));
    if (!Ufx || !Y || !ex || !bad) return 0;  // *bad_out stays null
    if (int rc = scratch_wait("bwd", st)) return rc;
    *bad_out = bad;
    const FxSmear P = fx_smear_params(rho, eps, 1.2);
    MCG_CK(cudaMemsetAsync(bad, 0, sizeof(unsigned), st));
    k_links_to_fx<<<blocks(nlinks, 128), 128, 0, st>>>((const double2*)U, Ufx, (size_t)g.vh, nlinks, bad);
    const unsigned nb = blocks(nlinks, 128);
    if (eps != 1.0) {
        k_smear_adjoint_fx<true><<<nb, 128, 0, st>>>(Ufx, (const double2*)Gout, Y, (int4*)Gin, ex, g, nfields, P, bad);
        k_smear_gather_fx<true><<<nb, 128, 0, st>>>(Ufx, Y, ex, (int4*)Gin, g, nfields, P, bad);
    } else {
        k_smear_adjoint_fx<false><<<nb, 128, 0, st>>>(Ufx, (const double2*)Gout, Y, (int4*)Gin, ex, g, nfields, P, bad);
        k_smear_gather_fx<false><<<nb, 128, 0, st>>>(Ufx, Y, ex, (int4*)Gin, g, nfields, P, bad);
    }
    MCG_CK(cudaGetLastError());
    note_launches(3);
    return 0;
}

// index-check counter of this unit (MCG_CHECK builds)
MCG_BOUND_READER(bound_hits_smear_bwd_fx)

}  // namespace mcg
