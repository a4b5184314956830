// The FP64 MCG half-sweep in fixed-point arithmetic (mcg_fx.cuh): links and
// transforms stay FP64 in memory, the site update runs on 64-bit integers.
//
// Inside the kernel link entries are integers of unit 2^-58 (|x| <= 1.03), the
// subgroup element's of unit 2^-60, A and b of the local problem (Sec. II.A: a
// site's share of R is a^T A a + 2 b.a + const on |a| = 1) of unit 2^-56, i.e.
// A / 16 and b / 16 in units of 2^-60.
#include <cuda_runtime.h>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"
#include "mcg_sweep.cuh"

namespace mcg {

// X 2^-60 as a float (X = h 2^32 + l)
__device__ __forceinline__ float fx_float_units(long long X) {  // in units of 2^-60
    const fx s = fx_split(X);
    return fmaf((float)s.h, 4294967296.f, (float)s.l);
}
// nearest integer of a float below 2^60 in magnitude
__device__ __forceinline__ long long float_to_ll(float v) {
    const int q = __float2int_rn(v * 0x1p-30f);
    return ((long long)q << 30) + __float2int_rn(fmaf(-(float)q, 0x1p30f, v));
}
// a float of magnitude below 7 in units of 2^-60
__device__ __forceinline__ long long float_to_fx(float v) {
    const float s = v * 0x1p28f;
    const int h = __float2int_rn(s);
    return ((long long)h << 32) + (long long)__float2int_rn((s - (float)h) * 0x1p31f) * 2;
}

// index of (k, j) in the packed upper triangle
__device__ __forceinline__ constexpr int tri(int k, int j) {
    return k <= j ? 4 * k - k * (k - 1) / 2 + j - k : 4 * j - j * (j - 1) / 2 + k - j;
}

struct Sol4 {
    long long a[4];
};

// Newton refinement of (a, mu) on the KKT system (mu - A) a = b, |a| = 1 from an
// FP32 seed: residuals in fixed point (exact to ~2^-57), corrections in FP32 by
// `inverse` (an FP32 inverse of mu - A), as kkt_refine_ldlt does with FP64
// residuals.  Stops once the correction is below 1e-12 (the next is below
// 1e-15) and normalises.  dmu: the multiplier's total change.  False if a
// correction is above 2^-6 or they do not get there in 8 steps.
template <class Inv>
__device__ __forceinline__ bool fx_refine(const fx (&A)[10], const long long (&b)[4], const float (&af)[4], float muf,
                                          const Inv& inverse, Sol4& r, float& dmu_total) {
    float y[4];
    inverse(af, y);
    const float inv_ay = __fdividef(1.f, af[0] * y[0] + af[1] * y[1] + af[2] * y[2] + af[3] * y[3]);
    long long mu = float_to_fx(muf);
#pragma unroll
    for (int k = 0; k < 4; ++k) r.a[k] = float_to_fx(af[k]);
    dmu_total = 0.f;
    bool ok = false;
    fx s[4];
#pragma unroll 1
    for (int it = 0; it < 8 && !ok; ++it) {
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = fx_split(r.a[k]);
        const fx m = fx_split(mu);
        float rf[4], x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            facc t = facc_zero();
            fx_msc(t, m, s[k]);
#pragma unroll
            for (int j = 0; j < 4; ++j) fx_mac(t, A[tri(k, j)], s[j]);
            rf[k] = fx_float_units(facc_get(t) + b[k]);
        }
        facc n = facc_zero();
#pragma unroll
        for (int k = 0; k < 4; ++k) fx_mac(n, s[k], s[k]);
        const float sres = 0.5f * fx_float_units((1LL << 60) - facc_get(n));
        inverse(rf, x);
        const float dmu = (af[0] * x[0] + af[1] * x[1] + af[2] * x[2] + af[3] * x[3] - sres) * inv_ay;
        float da[4], dmax = fabsf(dmu) * 0x1p-4f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            da[k] = fmaf(-dmu, y[k], x[k]);
            dmax = fmaxf(dmax, fabsf(da[k]));
        }
        if (!(dmax < 0x1p54f)) return false;  // NaN included: the seed is no use
#pragma unroll
        for (int k = 0; k < 4; ++k) r.a[k] += float_to_ll(da[k]);
        mu += float_to_ll(dmu);
        dmu_total += dmu;
        ok = dmax <= 1152921.5f;  // 1e-12
    }
    if (!ok) return false;
    dmu_total *= 0x1p-60f;
    // |a| = 1 to the last units: a (1 + (1 - |a|^2) / 2)
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = fx_split(r.a[k]);
    facc n = facc_zero();
#pragma unroll
    for (int k = 0; k < 4; ++k) fx_mac(n, s[k], s[k]);
    const float d = 0.5f * fx_float_units((1LL << 60) - facc_get(n));
#pragma unroll
    for (int k = 0; k < 4; ++k) r.a[k] += float_to_ll(af[k] * d);
    return true;
}

struct InvLdlt {
    const float (&L)[4][4];
    const float (&Dinv)[4];
    __device__ __forceinline__ void operator()(const float (&r)[4], float (&x)[4]) const { ldlt4_solve(L, Dinv, r, x); }
};
struct InvEigen {
    const float (&V)[4][4];
    const float (&d)[4];
    __device__ __forceinline__ void operator()(const float (&r)[4], float (&x)[4]) const {
        float t[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = (V[0][i] * r[0] + V[1][i] * r[1] + V[2][i] * r[2] + V[3][i] * r[3]) * d[i];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = V[k][0] * t[0] + V[k][1] * t[1] + V[k][2] * t[2] + V[k][3] * t[3];
    }
};

struct Prob {
    fx A[10];
    long long b[4];
};

// Seed for the problems whose maximum is far from e0 (most of an unfixed
// field's): Newton on 1 / |a(mu)| - 1 for the multiplier (Moré and Sorensen
// 1983), a(mu) = (mu - A)^-1 b, from mu = |A|_F + |b| above the root; a step
// that leaves mu - A indefinite is halved back towards the last definite one.
// True with mu, a and the factors of mu - A once | |a| - 1 | < 1e-3 (the
// refinement does the rest); false near the hard case.
__device__ __forceinline__ bool secular_ldlt(const float (&A)[4][4], const float (&b)[4], float (&a)[4], float& mu,
                                             float (&L)[4][4], float (&Dinv)[4], float& pd) {
    float f2 = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) f2 = fmaf(A[i][j], A[i][j], f2);
    mu = fsqrt(f2) + fsqrt(b[0] * b[0] + b[1] * b[1] + b[2] * b[2] + b[3] * b[3]);
    float good = mu;  // mu - A positive definite
#pragma unroll 1
    for (int it = 0; it < 16; ++it) {
        float M[4][4], y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) M[i][j] = (i == j ? mu : 0.f) - A[i][j];
        pd = ldlt4(M, L, Dinv);
        if (!(pd > 1e-6f)) {
            mu = 0.5f * (mu + good);
            continue;
        }
        good = mu;
        ldlt4_solve(L, Dinv, b, a);
        const float n2 = a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + a[3] * a[3];
        const float n = fsqrt(n2);
        if (fabsf(n - 1.f) < 1e-3f) return pd > 2e-4f;
        ldlt4_solve(L, Dinv, a, y);
        mu += __fdividef(n2 * (n - 1.f), a[0] * y[0] + a[1] * y[1] + a[2] * y[2] + a[3] * y[3]);
    }
    return false;
}

// The local problems neither seed settles: FP32 Jacobi + secular seed refined
// in fixed point, else the full FP64 Jacobi + secular solve.  Out of line; the
// problem is passed by value and the decomposition stays in registers (through
// memory a call took four times as long).
static __device__ __noinline__ Sol4 solve_fx_fallback(Prob p) {
    float Af[4][4], bf[4], af[4], muf, V[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        bf[i] = fx_float_units(p.b[i]) * 0x1p-60f;
#pragma unroll
        for (int j = 0; j < 4; ++j) Af[i][j] = fx_float_units(fx_join(p.A[tri(i, j)])) * 0x1p-60f;
    }
    Sol4 r;
    jacobi4<float>(Af, V, 8, 5e-7f);
    if (!trs_from_eigen<float>(Af, V, bf, af, muf)) {
        float amax = Af[0][0], amin = Af[0][0];
#pragma unroll
        for (int i = 1; i < 4; ++i) {
            amax = fmaxf(amax, Af[i][i]);
            amin = fminf(amin, Af[i][i]);
        }
        // the correction contracts by ~1e-7 of the spread over the gap mu -
        // lambda_max; the refined multiplier must stay above lambda_max by more
        // than the FP32 error of the eigenvalues
        const float gap = muf - amax, spread = muf - amin + 1e-30f;
        if (gap > 1e-5f * spread && muf < 7.f) {
            float d[4], dmu;
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = __fdividef(1.0f, muf - Af[i][i]);
            if (fx_refine(p.A, p.b, af, muf, InvEigen{V, d}, r, dmu) && gap + dmu > 3e-6f * spread) return r;
        }
    }
    double Ad[16], bd[4], ad[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        bd[i] = fx_double(p.b[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) Ad[4 * i + j] = fx_double(fx_join(p.A[tri(i, j)]));
    }
    solve_f64_full(Ad, bd, ad);
    const bool fin = isfinite(ad[0]) && isfinite(ad[1]) && isfinite(ad[2]) && isfinite(ad[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k)  // backstop: the identity leaves the site unchanged
        r.a[k] = fin ? fx_from_bits((unsigned long long)__double_as_longlong(ad[k])) : (k == 0 ? 1LL << 60 : 0LL);
    return r;
}

// Global maximum of the local problem; returns 1 when the warm-started path
// (FP32 Newton from a = e0, refined, certified above lambda_max) did not settle
// it.
__device__ __forceinline__ int solve_fx(const Prob& p, Sol4& r) {
    float Af[4][4], bf[4], af[4], muf;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        bf[i] = fx_float_units(p.b[i]) * 0x1p-60f;
#pragma unroll
        for (int j = i; j < 4; ++j)
            Af[i][j] = Af[j][i] = fmaf((float)p.A[tri(i, j)].l, 0x1p-60f, (float)p.A[tri(i, j)].h * 0x1p-28f);
    }
    float L[4][4], Dinv[4], pd, mu_f;
#pragma unroll 1
    for (int seed = 0; seed < 2; ++seed) {
        bool ok;
        if (seed == 0) {
            ok = kkt_newton<float>(Af, bf, af, muf, L, Dinv, pd, mu_f) && pd > 2e-4f;
        } else {
            ok = secular_ldlt(Af, bf, af, muf, L, Dinv, pd);
            mu_f = muf;
        }
        float dmu;
        if (ok && muf < 7.f && fx_refine(p.A, p.b, af, muf, InvLdlt{L, Dinv}, r, dmu)) {
            // above_lambda_max with margin 1e-6 (see mcg_sweep.cuh): the refined
            // multiplier against the det/trace bound of mu_f - A
            const float det = __fdividef(1.f, (Dinv[0] * Dinv[1]) * (Dinv[2] * Dinv[3]));
            const float tr = ((mu_f - Af[0][0]) + (mu_f - Af[1][1])) + ((mu_f - Af[2][2]) + (mu_f - Af[3][3]));
            if (((muf - mu_f) + dmu) + 27.f * __fdividef(det, tr * tr * tr) > 1e-6f * tr) return seed;
        }
    }
    r = solve_fx_fallback(p);
    return 1;
}

// rows 0 <- G rows for the SU(2) element a = (a0, a1, a2, a3) on rows xp, xq:
// (a0 + i a3) xp + (a2 + i a1) xq, (-a2 + i a1) xp + (a0 - i a3) xq.  Rounded (the
// sums start at one half) where the other products cut: a cut is a drift of half
// a unit per move in one direction, which after thousands of sweeps is more than
// all rounding (U against G U0 G^dag, 6 x 4 x 6 x 8 after 1 000 and 3 000 sweeps, rms:
// cut 9.2e-15 and 2.8e-14, rounded and stored as below 2.3e-15 and 5.4e-15, the FP64
// kernel 3.5e-15 and 6.6e-15).
__device__ __forceinline__ void fx_su2(const fx (&a)[4], fx na2, fx na3, cfx& xp, cfx& xq, long long rnd) {
    facc pr, pi, qr, qi;
    pr.hi = pi.hi = qr.hi = qi.hi = 0;
    pr.mid = pi.mid = qr.mid = qi.mid = rnd;
    fx_mac(pr, a[0], xp.re);
    fx_msc(pr, a[3], xp.im);
    fx_mac(pr, a[2], xq.re);
    fx_msc(pr, a[1], xq.im);
    fx_mac(pi, a[0], xp.im);
    fx_mac(pi, a[3], xp.re);
    fx_mac(pi, a[2], xq.im);
    fx_mac(pi, a[1], xq.re);
    fx_mac(qr, na2, xp.re);
    fx_msc(qr, a[1], xp.im);
    fx_mac(qr, a[0], xq.re);
    fx_mac(qr, a[3], xq.im);
    fx_mac(qi, na2, xp.im);
    fx_mac(qi, a[1], xp.re);
    fx_mac(qi, a[0], xq.im);
    fx_mac(qi, na3, xq.re);
    xp = cfx_get(pr, pi);
    xq = cfx_get(qr, qi);
}

// FP64 <-> integers of unit 2^-58; flip: the sign bit, to negate the imaginary part
__device__ __forceinline__ cfx load58(const double2* p, unsigned long long flip) {
    const double2 v = *p;
    cfx r;
    r.re = fx_split(fx_from_bits((unsigned long long)__double_as_longlong(v.x)) >> 2);
    r.im = fx_split(fx_from_bits((unsigned long long)__double_as_longlong(v.y) ^ flip) >> 2);
    return r;
}
__device__ __forceinline__ double double58(fx v, unsigned half) {
    return __longlong_as_double((long long)fx_to_bits(fx_join(v) * 4, half));
}

// Sum over the threads of a site (lanes SPW apart) of the raw accumulators: the
// same bits for every number of threads.
template <int SPW>
__device__ __forceinline__ long long fx_site_sum(facc v) {
#pragma unroll
    for (int o = SPW; o < 32; o *= 2) {
        v.hi += __shfl_xor_sync(0xffffffffu, v.hi, o);
        v.mid += __shfl_xor_sync(0xffffffffu, v.mid, o);
    }
    return facc_get(v);
}

// One half-sweep, TPS threads per site (a warp holds 32 / TPS sites, thread q
// of a site the q-th group of 8 / TPS of its links).  The backward links are
// held daggered, N = U_mu(x - mu)^dag, so that the move is rows P, Q of G M for
// all eight and their shares of A and b have one form.  A and b are summed over
// the site's threads by shuffles and every thread solves the local problem;
// integer sums make the result the same bits for every TPS.  A column (or two)
// of Omega(x) per thread stays in registers.
// Shared memory: 1152 / TPS bytes per thread, entry-major.
// CHECK (callers' fields that were not validated): a site whose matrices are
// not near-unitary (fx_bad_gram, or not finite) is left alone and marked in
// bt.left, which the FP64 kernel reads (by then the moved links' rows may have
// other norms).
// Bound by issue and the integer multiplier (52 % of the issue slots, of them a
// third multiply-adds), for small lattices by the latency of the three solves.
// Measured on 20^3 x 40: 285 us per half-sweep near a maximum (the FP64 kernel
// 917 us, FP64 pipe 82 %), 474 us on an unfixed field (1 100 us); 4^4: 16 us
// (98 us).
template <int TPS, int NT, int MINB, bool ACC, bool CHECK>
__global__ void __launch_bounds__(NT, MINB) k_halfsweep_fx(SweepBatch bt, int parity) {
    constexpr int NM = 8 / TPS, SPW = 32 / TPS;
    const double2 zero2 = make_double2(0.0, 0.0);
    extern __shared__ int4 fx_smem[];
    const int f = field_of_block(bt.desc, bt.nf, blockIdx.x);
    if (ACC) reunit_due(bt, f);
    if (bt.state[f].done) return;  // block-uniform
    const FieldDesc fd = bt.desc[f];
    const Geom g = fd.geo;
    double2* __restrict__ U = reinterpret_cast<double2*>(fd.U);
    double2* __restrict__ G = reinterpret_cast<double2*>(fd.G);
    const int lane = threadIdx.x & 31, q = lane / SPW;
    const int s = ((blockIdx.x - fd.blk0) * (NT / 32) + (threadIdx.x >> 5)) * SPW + lane % SPW;
    bool active = s < g.vh;
    int c[4];
    if (active) {
        eo_coords(g, parity, s, c);
        active = c[3] >= fd.t_lo && c[3] < fd.t_hi;  // the sites of a t-slab (whole lattice by default)
    }
    auto slot = [&](int i, int e) -> int4& { return fx_smem[(i * 9 + e) * NT + threadIdx.x]; };
    auto get = [&](int i, int e) {
        const int4 v = slot(i, e);
        cfx r;
        r.re.h = v.x;
        r.re.l = v.y;
        r.im.h = v.z;
        r.im.l = v.w;
        return r;
    };
    auto put = [&](int i, int e, cfx v) { slot(i, e) = make_int4(v.re.h, v.re.l, v.im.h, v.im.l); };
    // matrix i of this thread: its first entry, and the strides of rows and columns
    auto link = [&](int i, size_t& sr, size_t& sc) {
        const int l = q * NM + i, mu = l & 3;
        const bool back = l >= 4;
        const int sl = back ? eo_neighbor(g, c, mu, -1) : s;
        sr = (size_t)g.vh * (back ? 1 : 3);
        sc = (size_t)g.vh * (back ? 3 : 1);
        return U + lidx(g, mu, back ? parity ^ 1 : parity, 0, sl);
    };

    bool bad = false;
    if (active) {
        // all loads in flight at once, then converted in place
#pragma unroll 1
        for (int i = 0; i < NM; ++i) {
            size_t sr, sc;
            const double2* src = link(i, sr, sc);
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k) cp_async<16>(&slot(i, 3 * r + k), src + r * sr + k * sc);
            if (CHECK) bad = bad || fx_bad_matrix(src, sr, sc);
        }
        if (CHECK && q == 0) bad = bad || fx_bad_matrix(G + gidx(g, parity, 0, s), 3 * (size_t)g.vh, (size_t)g.vh);
        cp_async_wait_all();
#pragma unroll 1
        for (int i = 0; i < NM; ++i) {
            const unsigned long long flip = q * NM + i >= 4 ? 1ULL << 63 : 0;
#pragma unroll 1
            for (int r = 0; r < 9; r += 3)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    put(i, r + k, load58(reinterpret_cast<const double2*>(&slot(i, r + k)), flip));
        }
    }
    if (CHECK) {
        // the site is left to the FP64 kernel if any of its matrices is bad
        int b = bad;
#pragma unroll
        for (int o = SPW; o < 32; o *= 2) b |= __shfl_xor_sync(0xffffffffu, b, o);
        if (active && q == 0) {
            bt.left->site[s] = b != 0;
            if (b) atomicAdd(&bt.left->count, 1u);
        }
        active = active && !b;
    }

    // columns q, q + TPS of Omega(x)
    constexpr int NC = TPS == 2 ? 2 : 1;
    cfx w[NC][3];
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const double2 v = active && q + n * TPS < 3 ? G[gidx(g, parity, 3 * r + q + n * TPS, s)] : zero2;
            w[n][r] = load58(&v, 0);
        }
    int fb = 0;
    // one half of the moves' unit, kept in a register (as a literal it is moved there
    // for every sum: 0.7 % of a sweep)
    long long rnd = 1LL << 27;
    asm volatile("" : "+l"(rnd));
#pragma unroll 1
    for (int sg = 0; sg < 3; ++sg) {
        const int P = sg == 2 ? 1 : 0, Q = sg == 0 ? 1 : 2, R = 3 - P - Q;
        facc Aa[10], ba[4];
#pragma unroll
        for (int k = 0; k < 10; ++k) Aa[k] = facc_zero();
#pragma unroll
        for (int k = 0; k < 4; ++k) ba[k] = facc_zero();
        if (active) {
#pragma unroll 1
            for (int i = 0; i < NM; ++i) {
                const cfx m11 = get(i, 4 * P), m12 = get(i, 3 * P + Q), m21 = get(i, 3 * Q + P), m22 = get(i, 4 * Q);
                const cfx cc = get(i, 4 * R);
                // (m11 + m22, i (m21 + m12), m21 - m12, i (m11 - m22)), at most 2.06
                cfx v[4];
                v[0].re = fx_split(fx_join(m11.re) + fx_join(m22.re));
                v[0].im = fx_split(fx_join(m11.im) + fx_join(m22.im));
                v[1].re = fx_split(-fx_join(m21.im) - fx_join(m12.im));
                v[1].im = fx_split(fx_join(m21.re) + fx_join(m12.re));
                v[2].re = fx_split(fx_join(m21.re) - fx_join(m12.re));
                v[2].im = fx_split(fx_join(m21.im) - fx_join(m12.im));
                v[3].re = fx_split(fx_join(m22.im) - fx_join(m11.im));
                v[3].im = fx_split(fx_join(m11.re) - fx_join(m22.re));
                int t = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    fx_mac(ba[k], cc.re, v[k].re);
                    fx_mac(ba[k], cc.im, v[k].im);
#pragma unroll
                    for (int j = k; j < 4; ++j, ++t) {
                        fx_mac(Aa[t], v[k].re, v[j].re);
                        fx_mac(Aa[t], v[k].im, v[j].im);
                    }
                }
            }
        }
        Prob p;
#pragma unroll
        for (int k = 0; k < 10; ++k) p.A[k] = fx_split(fx_site_sum<SPW>(Aa[k]));
#pragma unroll
        for (int k = 0; k < 4; ++k) p.b[k] = fx_site_sum<SPW>(ba[k]);
        if (active) {
            Sol4 r;
            const int e = solve_fx(p, r);
            if (q == 0) fb += e;
            fx a[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) a[k] = fx_split(r.a[k]);
            const fx na2 = fx_neg(a[2]), na3 = fx_neg(a[3]);
#pragma unroll 1
            for (int i = 0; i < NM; ++i) {
#pragma unroll 1
                for (int k = 0; k < 3; ++k) {
                    cfx xp = get(i, 3 * P + k), xq = get(i, 3 * Q + k);
                    fx_su2(a, na2, na3, xp, xq, rnd);
                    put(i, 3 * P + k, xp);
                    put(i, 3 * Q + k, xq);
                }
            }
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                cfx xp = P == 0 ? w[n][0] : w[n][1], xq = Q == 1 ? w[n][1] : w[n][2];
                fx_su2(a, na2, na3, xp, xq, rnd);
                if (sg == 2) {
                    w[n][1] = xp;
                    w[n][2] = xq;
                } else {
                    w[n][0] = xp;
                    if (sg == 0) w[n][1] = xq;
                    if (sg == 1) w[n][2] = xq;
                }
            }
        }
    }

    facc tr2 = facc_zero();
    if (active) {
#pragma unroll 1
        for (int i = 0; i < NM; ++i) {
            size_t sr, sc;
            double2* dst = link(i, sr, sc);
            const unsigned long long flip = q * NM + i >= 4 ? 1ULL << 63 : 0;
            // ties (one entry in 32) away from zero as the forward link of its one end
            // and towards it as the backward link of the other: a link, stored by both
            // in turn, does not grow (ties to even cost 1.7 % of a sweep)
            const unsigned half = q * NM + i >= 4 ? 511u : 512u;
            long long tx = 0, ty = 0;
#pragma unroll 1
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const cfx v = get(i, 3 * r + k);
                    const unsigned long long im = fx_to_bits(fx_join(v.im) * 4, half) ^ flip;
                    dst[r * sr + k * sc] = make_double2(double58(v.re, half), __longlong_as_double((long long)im));
                    if (ACC && r == k) {
                        tx += fx_join(v.re);
                        ty += fx_join(v.im);
                    }
                }
            if (ACC) {
                const fx sx = fx_split(tx), sy = fx_split(ty);
                fx_mac(tr2, sx, sx);
                fx_mac(tr2, sy, sy);
            }
        }
#pragma unroll
        for (int n = 0; n < NC; ++n)
            if (q + n * TPS < 3) {
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    G[gidx(g, parity, 3 * r + q + n * TPS, s)] =
                        make_double2(double58(w[n][r].re, 512u), double58(w[n][r].im, 512u));
            }
    }
    if (ACC) {
        // a site's share (unit 2^-56, at most 72 (1.03)^2), cut to units of 2^-50, and
        // the sum over the warp's sites (below 2^61), as an integer: with the integer
        // sum of the partials R has the same bits for every number of threads per site
        long long r = fx_site_sum<SPW>(tr2) >> 6;
#pragma unroll
        for (int o = 1; o < SPW; o *= 2) r += __shfl_xor_sync(0xffffffffu, r, o);
        const int k = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
        if (lane == 0) {
            if (CHECK)
                bt.partial[k] = fx_double(r) * 0x1p10;
            else
                reinterpret_cast<long long*>(bt.partial)[k] = r;
        }
    }
    {
        const int w = __reduce_add_sync(0xffffffffu, fb);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(&bt.state[f].fallbacks, w);
    }
}

// Threads per site and block, by the number of sites of a parity (all fields
// that run side by side): more threads per site shorten a site's chain while
// the GPU is not full, fewer repeat the local solve less.  Measured, us per
// sweep for 2 / 4 / 8 threads: 128 sites 63 / 44 / 36, 2 048: 64 / 46 / 39,
// 5 040: 66 / 57 / 59, 10 368: 86 / 75 / 92, 19 208: 87 / 104 / 141, 160 000:
// 573 / 689 / 1 048.
FxShape fx_shape(long long sites) {
    if (sites <= 4096) return {8, 32};
    if (sites <= 16384) return {4, 64};
    return {2, 128};
}

template <int TPS, int NT, int MINB>
static int prepare_shape() {
    const int smem = 1152 / TPS * NT;
    MCG_CK(cudaFuncSetAttribute(k_halfsweep_fx<TPS, NT, MINB, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    MCG_CK(cudaFuncSetAttribute(k_halfsweep_fx<TPS, NT, MINB, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return 0;
}
int prepare_halfsweep_fx() {
    int rc = 0;
    if ((rc = prepare_shape<2, 128, 3>()) || (rc = prepare_shape<4, 64, 6>()) || (rc = prepare_shape<8, 32, 12>()))
        return rc;
    const int smem = 1152 / 2 * 128;
    MCG_CK(cudaFuncSetAttribute(k_halfsweep_fx<2, 128, 3, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    MCG_CK(cudaFuncSetAttribute(k_halfsweep_fx<2, 128, 3, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return 0;
}

template <int TPS, int NT, int MINB>
static void launch_shape(bool acc, const SweepBatch& bt, int parity, int nblocks, cudaStream_t st) {
    const size_t smem = 1152 / TPS * NT;
    if (acc)
        k_halfsweep_fx<TPS, NT, MINB, true, false><<<nblocks, NT, smem, st>>>(bt, parity);
    else
        k_halfsweep_fx<TPS, NT, MINB, false, false><<<nblocks, NT, smem, st>>>(bt, parity);
}
void launch_halfsweep_fx(FxShape sh, bool acc, const SweepBatch& bt, int parity, int nblocks, cudaStream_t st) {
    if (bt.left) {  // unvalidated fields: shape (2, 128)
        const size_t smem = 1152 / 2 * 128;
        if (acc)
            k_halfsweep_fx<2, 128, 3, true, true><<<nblocks, 128, smem, st>>>(bt, parity);
        else
            k_halfsweep_fx<2, 128, 3, false, true><<<nblocks, 128, smem, st>>>(bt, parity);
    } else if (sh.tps == 8) {
        launch_shape<8, 32, 12>(acc, bt, parity, nblocks, st);
    } else if (sh.tps == 4) {
        launch_shape<4, 64, 6>(acc, bt, parity, nblocks, st);
    } else {
        launch_shape<2, 128, 3>(acc, bt, parity, nblocks, st);
    }
}

// index-check counter of this unit (MCG_CHECK builds)
MCG_BOUND_READER(bound_hits_sweep_fx)

}  // namespace mcg
