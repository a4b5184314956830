// FP64 smearing in fixed-point arithmetic (mcg_fx.cuh): the step of
// mcg_smear.cu on fields held as 64-bit integers of unit 2^-60.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"
#include "mcg_smear_fx.cuh"

namespace mcg {

// ---------------------------------------------------------------------------
// Products that neighbouring links share, from a first pass over ordered pairs of
// directions (a, b) and sites y: the corner K_ab(y) = U_a(y) U_b(y+a) and, for
// over-improved steps, the two plaquette staples that it closes,
// P_ab(y) = K_ab(y) U_a(y+b)^dag (from y to y + b) and D_ab(y) = U_b(y)^dag K_ab(y)
// (from y + b to y + b + a).
// Stout: 3 products per link for the corners, then one per staple: 11 with the
// step's own two instead of 14.  Over-improved: 9 per link, then the plaquette
// staples are loads and the 18 rectangles take 30 products: 41 instead of 86.
// (Storing the other two corners of a plaquette as well would make 38, for a
// third more memory.)  12 or 36 matrices per site: 1 728 or 5 184 bytes.
// Measured, ms per step with this pass, without and with the products: stout on
// 20^3 x 40 0.93 and 0.89 (0.81 tiled), on 16^4 0.198 and 0.191; over-improved on
// 12 x 10 x 14 x 22 0.63 and 0.37.
// ---------------------------------------------------------------------------
template <bool RECT>
constexpr int kFxAux = RECT ? 36 : 12;  // matrices per site: the 12 K, then the P, then the D
__device__ __forceinline__ int fx_pair(int a, int b) { return 3 * a + (b < a ? b : b - 1); }

__device__ __forceinline__ size_t fx_aux_idx(const Geom& g, int slot, int p, int s) {
#ifdef MCG_CHECK
    if (mcg_bad((unsigned)slot >= (unsigned)kFxAux<true> || (unsigned)p >= 2u || (unsigned)s >= (unsigned)g.vh)) return 0;
#endif
    return ((size_t)(2 * slot + p) * 9) * g.vh + s;
}

// A factor of a path: kind 0 / 1: the link of direction mu / nu, 2 / 3: K_numu /
// K_munu, 4 / 5: P, 6 / 7: D; displacement (dm, dn) of its site from x, daggered
// or not
struct FxAuxFactor {
    signed char kind, dm, dn, dag;
};
// the shapes of c_fx_paths in their order
__constant__ FxAuxFactor c_fx_aux_paths[10][3] = {
    {{4, 0, 0, 0}, {0, 0, 0, 0}, {0, 0, 0, 0}},
    {{7, 0, -1, 0}, {0, 0, 0, 0}, {0, 0, 0, 0}},
    {{1, 0, 0, 0}, {4, 0, 1, 0}, {1, 1, 0, 1}},
    {{1, 0, -1, 1}, {7, 0, -2, 0}, {1, 1, -1, 0}},
    {{2, 0, 0, 0}, {5, 1, 0, 1}, {0, 0, 0, 0}},
    {{1, 0, -1, 1}, {0, 0, -1, 0}, {5, 1, -1, 0}},
    {{6, -1, 0, 0}, {0, 0, 1, 0}, {1, 1, 0, 1}},
    {{6, -1, -1, 1}, {3, 0, -1, 0}, {0, 0, 0, 0}},
    // plaquettes from the corners alone
    {{2, 0, 0, 0}, {1, 1, 0, 1}, {0, 0, 0, 0}},
    {{1, 0, -1, 1}, {3, 0, -1, 0}, {0, 0, 0, 0}},
};
__constant__ signed char c_fx_aux_len[10] = {1, 1, 3, 3, 2, 3, 3, 2, 2, 2};

__device__ __forceinline__ void fx_aux_factor(const int4* __restrict__ U, const int4* __restrict__ A, const Geom& g,
                                              const int c[4], int mu, int nu, FxAuxFactor f, cfx* m) {
    int q[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const int v = c[d] + (d == mu ? f.dm : 0) + (d == nu ? f.dn : 0);
        q[d] = v < 0 ? v + g.n[d] : (v >= g.n[d] ? v - g.n[d] : v);
    }
    const int p = (q[0] + q[1] + q[2] + q[3]) & 1;
    const int s = eo_index(g, q);
    const int4* base = f.kind < 2 ? U + lidx(g, f.kind ? nu : mu, p, 0, s)
                                  : A + fx_aux_idx(g, 12 * ((f.kind >> 1) - 1) +
                                                          ((f.kind & 1) ? fx_pair(mu, nu) : fx_pair(nu, mu)), p, s);
    fx_load_entries(base, (size_t)g.vh, f.dag, m);
}

// fx_staple_sum from the first pass's products
template <bool RECT>
__device__ __forceinline__ void fx_staple_sum_shared(const int4* __restrict__ U, const int4* __restrict__ A,
                                                  const Geom& g, const int c[4], int mu, const FxSmear& P, cfx* a,
                                                  cfx* b) {
    long long C[18];
#pragma unroll
    for (int e = 0; e < 18; ++e) C[e] = 0;
#pragma unroll 1
    for (int k = RECT ? 7 : 9; k >= (RECT ? 0 : 8); --k) {
        const int nf = RECT ? c_fx_aux_len[k] : 2;
        if (RECT && k == 1) {
#pragma unroll
            for (int e = 0; e < 18; ++e) C[e] = fx_mul(fx_split(C[e]), P.wr);
        }
#pragma unroll 1
        for (int nu = 0; nu < 4; ++nu) {
            if (nu == mu) continue;
            fx_aux_factor(U, A, g, c, mu, nu, c_fx_aux_paths[k][0], a);
#pragma unroll 1
            for (int j = 1; j < nf; ++j) {
                fx_aux_factor(U, A, g, c, mu, nu, c_fx_aux_paths[k][j], b);
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

// the first pass: thread per (field, site, parity, pair)
template <bool RECT>
__global__ void __launch_bounds__(128, 3) k_smear_products_fx(const int4* __restrict__ Uin, int4* __restrict__ Aux,
                                                              Geom g, int nfields) {
    LinkItem it;
    if (!(!RECT && link_tiled(g) ? link_item<true>(g, 12, nfields, it) : link_item<false>(g, 12, nfields, it))) return;
    const int f = it.f, p = it.p, s = it.s, pair = it.kind;
    const int da = pair / 3, pb = pair - 3 * da, db = pb < da ? pb : pb + 1;
    const size_t vh = (size_t)g.vh;
    const int4* U = Uin + (size_t)f * link_elems(g);
    int4* out = Aux + (size_t)f * (kFxAux<RECT> / 4) * link_elems(g) + fx_aux_idx(g, pair, p, s);
    const size_t kind = 12 * 18 * vh;  // from one kind of product to the next
    int c[4];
    eo_coords(g, p, s, c);
    const int sa = eo_neighbor(g, c, da, +1), sb = eo_neighbor(g, c, db, +1);
    cfx K[9], a[9], b[9];
    fx_load_entries(U + lidx(g, da, p, 0, s), vh, false, K);
    fx_load_entries(U + lidx(g, db, p ^ 1, 0, sa), vh, false, b);
    m3fx_mul_inplace<false>(K, b);
#pragma unroll
    for (int e = 0; e < 9; ++e) out[e * vh] = fx_pack(K[e]);
    if (!RECT) return;
    fx_load_entries(U + lidx(g, da, p ^ 1, 0, sb), vh, true, b);
#pragma unroll
    for (int e = 0; e < 9; ++e) a[e] = K[e];
    m3fx_mul_inplace<false>(a, b);
#pragma unroll
    for (int e = 0; e < 9; ++e) out[kind + e * vh] = fx_pack(a[e]);
    fx_load_entries(U + lidx(g, db, p, 0, s), vh, true, a);
    m3fx_mul_inplace<false>(a, K);
#pragma unroll
    for (int e = 0; e < 9; ++e) out[2 * kind + e * vh] = fx_pack(a[e]);
}

// exp(iQ) with Q = 2 x, x traceless Hermitian of spectral radius at most 0.67.
// Powers of x reduce by Cayley-Hamilton, x^3 = c1 x + c0:
// x^k = a_k + b_k x + b_{k-1} x^2 with a_k = c0 b_{k-2} and
// b_{k+1} = c1 b_{k-1} + c0 b_{k-2}, so
// exp(iQ) = sum_k (2^k / k!) i^k x^k = f0 + f1 x + f2 x^2 needs one three-term
// recurrence of reals.  (No square root, division or angle, and no case near
// degenerate eigenvalues.)
__device__ __forceinline__ void fx_exp(const fx (&d)[3], const cfx (&x)[3], const FxSmear& P, cfx* E) {
    fx c0, c1, y[3];
    fx_invariants(d, x, c0, c1, y);
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
        fx_mac(s, c1, b1);
        fx_mac(s, c0, b2);
        fx n = fx_split(facc_get(s));
        fx_mac(f1i, to, n);
        fx_mac(f2i, to, b);
        fx_mac(gi, to, b1);
        s = facc_zero();
        fx_mac(s, c1, b);
        fx_mac(s, c0, b1);
        b2 = b;
        b1 = n;
        b = fx_split(facc_get(s));
    }
    const cfx f1 = cfx_get(f1r, f1i), f2 = cfx_get(f2r, f2i);
    cfx f0;
    f0.re = fx_split(fx_mul(fx_split(facc_get(gr)), c0) + (1LL << 60));
    f0.im = fx_split(fx_mul(fx_split(facc_get(gi)), c0));
    fx_exp_matrix(d, x, y, f0, f1, f2, E);
}

// One thread per link, old field in, new field out (fixed point, or FP64 after
// the last step).
// Bound by the integer multiplier.  Measured on 20^3 x 40, first pass included:
// 0.81 ms per stout step (the FP64 kernel: 4.88 ms, FP64 pipe 93 % busy);
// over-improved steps on 12 x 10 x 14 x 22: 0.37 ms (2.70 ms).  3 blocks of 128
// per SM: 2 blocks take 12 %, 4 (spilling) 4 % longer.  Deviation from a 128-bit reference (4^4, ten
// stout steps): 8.5e-17 rms, the FP64 kernel's 2.2e-16.
template <bool RECT, bool SHARED, bool OUT64>
__global__ void __launch_bounds__(128, 3) k_smear_step_fx(const int4* __restrict__ Uin, const int4* __restrict__ Aux,
                                                          int4* __restrict__ Uout, Geom g, int nfields,
                                                          const __grid_constant__ FxSmear P) {
    int f, mu, p, s;
    if (RECT) {  // link_item<false> without whole warps, which the step took 0.8 % longer with
        const long long n = 8LL * g.vh * nfields;
        const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (id >= n) return;
        f = (int)(id / (8LL * g.vh));
        int r = (int)(id - (long long)f * 8 * g.vh);
        mu = r / (2 * g.vh);
        r -= mu * 2 * g.vh;
        p = r / g.vh;
        s = r - p * g.vh;
    } else {
        LinkItem it;
        if (!(link_tiled(g) ? link_item<true>(g, 4, nfields, it) : link_item<false>(g, 4, nfields, it))) return;
        f = it.f;
        mu = it.kind;
        p = it.p;
        s = it.s;
    }
    const int4* U = Uin + (size_t)f * link_elems(g);
    int c[4];
    eo_coords(g, p, s, c);

    cfx a[9], b[9];
    if (SHARED)
        fx_staple_sum_shared<RECT>(U, Aux + (size_t)f * (kFxAux<RECT> / 4) * link_elems(g), g, c, mu, P, a, b);
    else
        fx_staple_sum<RECT>(U, g, c, mu, P, a, b);
    const int4* ul = U + lidx(g, mu, p, 0, s);
#pragma unroll
    for (int e = 0; e < 9; ++e) b[e] = fx_load(ul + (size_t)e * g.vh);
    m3fx_mul_inplace<true>(a, b);  // Omega = C U^dag
    fx d[3];
    cfx x[3];
    fx_generator(a, P.third, d, x);
    fx_exp(d, x, P, a);
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

__global__ void __launch_bounds__(256) k_to_fx(const double2* __restrict__ src, int4* __restrict__ dst, size_t n) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double2 v = src[k];
    cfx r;
    r.re = fx_of(v.x);
    r.im = fx_of(v.y);
    dst[k] = fx_pack(r);
}

void launch_to_fx(const void* src, void* dst, size_t n, cudaStream_t st) {
    k_to_fx<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double2*)src, (int4*)dst, n);
}

bool smear_fx_applies(double rho, double eps) {
    const double cp = (5.0 - 2.0 * eps) / 3.0, cr = -(1.0 - eps) / 12.0;
    return std::fabs(rho) * (6.0 * std::fabs(cp) + 18.0 * std::fabs(cr)) <= 1.0;
}

static fx host_fx(double v) { return fx_split(std::llrint(std::ldexp(v, 60))); }

FxSmear fx_smear_params(double rho, double eps, double slack) {
    const double cp = (5.0 - 2.0 * eps) / 3.0, cr = -(1.0 - eps) / 12.0;
    FxSmear P;
    P.wp = host_fx(rho * cp);
    P.wr = host_fx(8.0 * rho * cr);
    const double weight = std::fabs(rho) * (6.0 * std::fabs(cp) + 18.0 * std::fabs(cr));
    P.gs = weight > 0.0 ? -std::ilogb(weight) - 1 : 0;
    if (P.gs < 0) P.gs = 0;  // weight = 1
    P.gp = host_fx(std::ldexp(rho * cp, P.gs));
    P.gr64 = host_fx(std::ldexp(64.0 * rho * cr, P.gs));
    P.third = fx_split(((1LL << 60) + 1) / 3);
    // 2^k / k! with 40 guard bits, rounded to 2^-60; terms until the bound
    // r^k / k! on the rest is below 2^-62, r = 4/3 of the staple weight
    const double rad = slack * 4.0 / 3.0 * weight;
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
    return P;
}

template <bool RECT, bool SHARED>
static auto step_kernel(bool out64) {
    return out64 ? k_smear_step_fx<RECT, SHARED, true> : k_smear_step_fx<RECT, SHARED, false>;
}
static auto step_kernel(bool rect, bool shared, bool out64) {
    return rect ? (shared ? step_kernel<true, true>(out64) : step_kernel<true, false>(out64))
                : (shared ? step_kernel<false, true>(out64) : step_kernel<false, false>(out64));
}

// Scratch of the products at most: 9.9 million sites of a stout step, 3.3 million
// of an over-improved one at a time, and fewer fields at a time where a quarter of
// the free memory is less.  A field beyond that takes the step that multiplies
// every path out.
constexpr size_t kFxAuxBytes = (size_t)16 << 30;

int run_smear_fx(const void* Uin, void* Uout, const Geom& g, int nfields, double rho, double eps, int n, bool* ran,
                 cudaStream_t st) {
    const size_t elems = link_elems(g) * (size_t)nfields;
    // several steps need a second field in any arithmetic, one step only here
    int rc = 0;
    void* tmp = n >= 2 ? scratch_device("smear.tmp", 16 * elems, &rc) : scratch_device_optional("smear.tmp", 16 * elems);
    if (rc) return rc;
    *ran = tmp != nullptr;
    if (!tmp) return 0;
    if ((rc = scratch_wait("smear", st))) return rc;
    const bool rect = eps != 1.0;
    const FxSmear P = fx_smear_params(rho, eps, 1.0);
    const bool tiled = !rect && link_tiled(g);
    // step k's source: tmp or Uout in turn, so that the last step reads tmp
    auto buf = [&](int k) { return (n - 1 - k) % 2 == 0 ? tmp : Uout; };
    launch_to_fx(Uin, buf(0), elems, st);
    // fields per pass: all, or as many as the products' scratch has room for
    int chunk = nfields;
    int4* aux = nullptr;
    const size_t per_field = 16 * ((rect ? kFxAux<true> : kFxAux<false>) / 4) * link_elems(g);
    chunk = (int)std::min<size_t>(nfields, kFxAuxBytes / per_field);
    if (chunk > 0) aux = (int4*)scratch_device_optional("smear.products", per_field * chunk);
    if (chunk > 0 && !aux) {
        chunk = (int)std::min<size_t>(chunk, scratch_optional_room("smear.products") / per_field);
        if (chunk > 0) aux = (int4*)scratch_device_optional("smear.products", per_field * chunk);
    }
    if (!aux) chunk = nfields;
    for (int k = 0; k < n; ++k) {
        const bool last = k + 1 == n;
        for (int f0 = 0; f0 < nfields; f0 += chunk) {
            const int nf = std::min(chunk, nfields - f0);
            const size_t off = (size_t)f0 * link_elems(g);
            const int4* src = (const int4*)buf(k) + off;
            int4* dst = (int4*)(last ? Uout : buf(k + 1)) + off;
            if (aux) {
                (rect ? k_smear_products_fx<true> : k_smear_products_fx<false>)
                    <<<link_blocks(tiled, g, 12, nf), 128, 0, st>>>(src, aux, g, nf);
                note_launches(1);
            }
            const auto step = step_kernel(rect, aux != nullptr, last);
            const unsigned nb = rect ? (unsigned)((8LL * g.vh * nf + 127) / 128) : link_blocks(tiled, g, 4, nf);
            step<<<nb, 128, 0, st>>>(src, aux, dst, g, nf, P);
            note_launches(1);
        }
    }
    MCG_CK(cudaGetLastError());
    note_launches(1);
    return scratch_mark("smear", st);
}

// index-check counter of this unit (MCG_CHECK builds)
MCG_BOUND_READER(bound_hits_smear_fx)

}  // namespace mcg
