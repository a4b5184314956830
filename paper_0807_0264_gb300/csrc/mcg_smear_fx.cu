// FP64 smearing in fixed-point arithmetic (mcg_fx.cuh): the step of
// mcg_smear.cu on fields held as 64-bit integers of unit 2^-60.
#include <cuda_runtime.h>

#include <cmath>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"
#include "mcg_smear_fx.cuh"

namespace mcg {

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

    cfx a[9], b[9];
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
    P.wr64 = host_fx(64.0 * rho * cr);
    P.third = fx_split(((1LL << 60) + 1) / 3);
    // 2^k / k! with 40 guard bits, rounded to 2^-60; terms until the bound
    // r^k / k! on the rest is below 2^-62, r = 4/3 of the staple weight
    const double rad = slack * 4.0 / 3.0 * std::fabs(rho) * (6.0 * std::fabs(cp) + 18.0 * std::fabs(cr));
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

int run_smear_fx(const void* Uin, void* Uout, const Geom& g, int nfields, double rho, double eps, int n,
                 cudaStream_t st) {
    const size_t elems = link_elems(g) * (size_t)nfields;
    int rc = 0;
    void* tmp = scratch_device("smear.tmp", 16 * elems, &rc);
    if (rc) return rc;
    const bool rect = eps != 1.0;
    const FxSmear P = fx_smear_params(rho, eps, 1.0);
    // step k's source: tmp or Uout in turn, so that the last step reads tmp
    auto buf = [&](int k) { return (n - 1 - k) % 2 == 0 ? tmp : Uout; };
    launch_to_fx(Uin, buf(0), elems, st);
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
