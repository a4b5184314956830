// Field kernels in fixed-point arithmetic (mcg_fx.cuh): gauge transforms of FP64
// fields, the mixed-precision hand-off and the plaquette.  Fields of these entry
// points are not always validated: a thread that meets a matrix with an entry or a
// row norm out of range does its link or plaquette in FP64.
//
// A transformed field that later sweeps round to FP32 keeps the FP64 kernels of
// mcg_field.cu: one entry rounded the other way moved the links of an unfixed
// 20^3 x 40 field by 1.4e-7 after 150 over-relaxed FP32 sweeps, and a link by
// 3e-8 in the double-float sweeps, whose local problems are built from the FP32
// parts; so those results stay what they were.
#include <cuda_runtime.h>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"

namespace mcg {

namespace {

template <typename T>
struct Vec2;
template <>
struct Vec2<double> {
    typedef double2 type;
};
template <>
struct Vec2<float> {
    typedef float2 type;
};

inline unsigned blocks(long long n, int nt) { return (unsigned)((n + nt - 1) / nt); }

// ---- gauge transform: U_mu(x) <- Omega(x) U_mu(x) Omega(x+mu)^dag ----------------
__device__ __noinline__ void apply_link_f64(double2* u, const double2* w, const double2* wf, size_t vh) {
    cplx<double> a[9], b[9], t[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        a[e] = mk(w[e * vh].x, w[e * vh].y);
        b[e] = mk(u[e * vh].x, u[e * vh].y);
    }
    m3_mul(a, b, t);
#pragma unroll
    for (int e = 0; e < 9; ++e) b[e] = mk(wf[e * vh].x, wf[e * vh].y);
    m3_mul_nd(t, b, a);
#pragma unroll
    for (int e = 0; e < 9; ++e) u[e * vh] = make_double2(a[e].x, a[e].y);
}

// A site whose transform the hand-off did not take in fixed point: no low half has
// this value (fx_split)
constexpr int kFxMarked = -0x7fffffff - 1;

// The compact FP32 (or hi + lo) transform of a site, re-unitarised in FP64
__device__ __forceinline__ void handoff_transform_f64(const float4* W, const float4* Wlo, size_t vh, cplx<double>* w) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float4 v = W[q * vh], l = Wlo ? Wlo[q * vh] : make_float4(0.f, 0.f, 0.f, 0.f);
        w[2 * q] = mk((double)v.x + (double)l.x, (double)v.y + (double)l.y);
        w[2 * q + 1] = mk((double)v.z + (double)l.z, (double)v.w + (double)l.w);
    }
#pragma unroll
    for (int e = 6; e < 9; ++e) w[e] = mk(0.0, 0.0);
    m3_reunitarise(w);
}
// u <- w u wf^dag in FP64 where one of the transforms is marked
__device__ __noinline__ void handoff_link_f64(double2* u, const int4* w, const int4* wf, const float4* W,
                                              const float4* Wlo, const float4* Wf, const float4* Wflo, size_t vh) {
    cplx<double> a[9], b[9], t[9];
    auto transform = [&](const int4* x, const float4* hi, const float4* lo, cplx<double>* m) {
        if (x->y == kFxMarked) {
            handoff_transform_f64(hi, lo, vh, m);
            return;
        }
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const cfx v = fx_load(x + e * vh);
            m[e] = mk(fx_double(fx_join(v.re)), fx_double(fx_join(v.im)));
        }
    };
    transform(w, W, Wlo, a);
#pragma unroll
    for (int e = 0; e < 9; ++e) b[e] = mk(u[e * vh].x, u[e * vh].y);
    m3_mul(a, b, t);
    transform(wf, Wf, Wflo, b);
    m3_mul_nd(t, b, a);
#pragma unroll
    for (int e = 0; e < 9; ++e) u[e * vh] = make_double2(a[e].x, a[e].y);
}

// One thread per link.  WFX: the transform in fixed point, of an SU(3) field (the
// hand-off; W and Wlo are what it came from, read for marked sites).  Two products
// and 18 to 54 conversions per link, bound by the integer multiplier.  A thread
// per link: the products need no more registers than three blocks of 128 per SM
// leave, and small lattices fill more SMs.
template <bool WFX>
__global__ void __launch_bounds__(128, 3) k_apply_gauge_fx(double2* Uall, const void* Gall, const float4* W,
                                                           const float4* Wlo, Geom g, int nfields) {
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= 8LL * g.vh * nfields) return;
    const int f = (int)(id / (8LL * g.vh));
    int r = (int)(id - (long long)f * 8 * g.vh);
    const int mu = r / (2 * g.vh);
    r -= mu * 2 * g.vh;
    const int p = r / g.vh, s = r - p * g.vh;
    const size_t vh = (size_t)g.vh;
    int c[4];
    eo_coords(g, p, s, c);
    const size_t iw = (size_t)f * gauge_elems(g) + gidx(g, p, 0, s);
    const int sf = eo_neighbor(g, c, mu, +1);
    const size_t iwf = (size_t)f * gauge_elems(g) + gidx(g, p ^ 1, 0, sf);
    double2* u = Uall + (size_t)f * link_elems(g) + lidx(g, mu, p, 0, s);
    cfx a[9], b[9];
    bool bad = false;
    if (WFX) {
        const int4* w = reinterpret_cast<const int4*>(Gall) + iw;
#pragma unroll
        for (int e = 0; e < 9; ++e) a[e] = fx_load(w + e * vh);
        bad = a[0].re.l == kFxMarked;
    } else {
        bad = fx_load_matrix(reinterpret_cast<const double2*>(Gall) + iw, 3 * vh, vh, a);
    }
    const bool ubad = fx_load_matrix(u, 3 * vh, vh, b);
    if (!WFX) bad = bad || ubad;
    m3fx_mul_inplace<false>(a, b);
    if (WFX) {
        const int4* w = reinterpret_cast<const int4*>(Gall) + iwf;
#pragma unroll
        for (int e = 0; e < 9; ++e) b[e] = fx_load(w + e * vh);
        bad = bad || b[0].re.l == kFxMarked;
    } else {
        bad = fx_load_matrix(reinterpret_cast<const double2*>(Gall) + iwf, 3 * vh, vh, b) || bad;
    }
    if (!WFX && bad) {
        apply_link_f64(u, reinterpret_cast<const double2*>(Gall) + iw, reinterpret_cast<const double2*>(Gall) + iwf, vh);
        return;
    }
    m3fx_mul_inplace<true>(a, b);
    if (WFX && bad) {
        const size_t i = (size_t)f * c12_gauge_chunks(g) + c12_gidx(g, p, 0, s);
        const size_t j = (size_t)f * c12_gauge_chunks(g) + c12_gidx(g, p ^ 1, 0, sf);
        handoff_link_f64(u, reinterpret_cast<const int4*>(Gall) + iw, reinterpret_cast<const int4*>(Gall) + iwf, W + i,
                         Wlo ? Wlo + i : nullptr, W + j, Wlo ? Wlo + j : nullptr, vh);
        return;
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) fx_store(u + e * vh, a[e]);
}

// ---- hand-off of the mixed schedule, pass 1 --------------------------------------
// W (compact: rows 0 and 1, FP32 or hi + lo) re-unitarised, to scratch in fixed
// point; Omega <- reunit(W Omega).  Omega is a validated transform, W unitary to
// FP32 rounding: a site where it is not (or not finite) is marked for pass 2 and
// done in FP64.  The marks are looked at behind the products of both passes: with
// the branches ahead, the loads behind them waited (both passes on 20^3 x 40, hi and
// hi + lo: 229 and 237 us, 232 and 241 with the branches ahead, 227 and 236 without
// any mark).
__device__ __noinline__ void handoff_gauge_f64(const float4* W, const float4* Wlo, double2* G, size_t vh) {
    cplx<double> w[9], o[9], t[9];
    handoff_transform_f64(W, Wlo, vh, w);
#pragma unroll
    for (int e = 0; e < 9; ++e) o[e] = mk(G[e * vh].x, G[e * vh].y);
    m3_mul(w, o, t);
    m3_reunitarise(t);
#pragma unroll
    for (int e = 0; e < 9; ++e) G[e * vh] = make_double2(t[e].x, t[e].y);
}
__global__ void __launch_bounds__(128, 3) k_handoff_gauge_fx(const float4* __restrict__ W,
                                                              const float4* __restrict__ Wlo, int4* __restrict__ Wfx,
                                                              double2* __restrict__ G, Geom g, int nfields) {
    const long long n = 2LL * g.vh * nfields;
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= n) return;
    const int f = (int)(id / (2LL * g.vh));
    const int r = (int)(id - (long long)f * 2 * g.vh);
    const int p = r / g.vh, s = r - p * g.vh;
    const size_t off = (size_t)f * gauge_elems(g) + gidx(g, p, 0, s), vh = (size_t)g.vh;
    const size_t coff = (size_t)f * c12_gauge_chunks(g) + c12_gidx(g, p, 0, s);
    cfx w[9], o[9];
    float size = 0.f;  // squared norm of rows 0 and 1, 2 for a unitary W (NaN fails the test)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float4 v = W[coff + q * vh];
        size = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, size))));
        w[2 * q].re = fx_of(v.x);
        w[2 * q].im = fx_of(v.y);
        w[2 * q + 1].re = fx_of(v.z);
        w[2 * q + 1].im = fx_of(v.w);
        if (Wlo) {
            const float4 l = Wlo[coff + q * vh];
            size = fmaf(l.x, l.x, fmaf(l.y, l.y, fmaf(l.z, l.z, fmaf(l.w, l.w, size))));
            w[2 * q].re = fx_split(fx_join(w[2 * q].re) + fx_join(fx_of(l.x)));
            w[2 * q].im = fx_split(fx_join(w[2 * q].im) + fx_join(fx_of(l.y)));
            w[2 * q + 1].re = fx_split(fx_join(w[2 * q + 1].re) + fx_join(fx_of(l.z)));
            w[2 * q + 1].im = fx_split(fx_join(w[2 * q + 1].im) + fx_join(fx_of(l.w)));
        }
    }
    const bool bad = m3fx_reunitarise(w) || !(size < 2.1f);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        Wfx[off + e * vh] = e == 0 && bad ? make_int4(0, kFxMarked, 0, 0) : fx_pack(w[e]);
        const double2 v = G[off + e * vh];
        o[e].re = fx_of(v.x);
        o[e].im = fx_of(v.y);
    }
    m3fx_mul_inplace<false>(w, o);
    m3fx_reunitarise(w);
    if (bad) {  // not before the loads of Omega, which would wait for the branch
        handoff_gauge_f64(W + coff, Wlo ? Wlo + coff : nullptr, G + off, vh);
        return;
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) fx_store(G + off + e * vh, w[e]);
}

// ---- plaquette -------------------------------------------------------------------
template <typename V>
__device__ __noinline__ double plaquette_f64(const V* a, const V* b, const V* c, const V* d, size_t vh) {
    cplx<double> x[9], y[9], t[9], q[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        x[e] = mk((double)a[e * vh].x, (double)a[e * vh].y);
        y[e] = mk((double)b[e * vh].x, (double)b[e * vh].y);
    }
    m3_mul(x, y, t);
#pragma unroll
    for (int e = 0; e < 9; ++e) y[e] = mk((double)c[e * vh].x, (double)c[e * vh].y);
    m3_mul_nd(t, y, q);
    double tr = 0.0;
#pragma unroll
    for (int e = 0; e < 9; ++e) tr += q[e].x * (double)d[e * vh].x + q[e].y * (double)d[e * vh].y;
    return tr;
}

// Per-block partial of the sum over sites of (1/3) Re tr of the six plaquettes:
// X = U_mu(x) U_nu(x+mu) and Y = U_nu(x) U_mu(x+nu) row by row, sum Re X Y^*.
// Two threads per site, three planes each (mu = 0; mu = 1 and 2), 2 bpf blocks of
// 128 sites per field: the six planes of a site are a serial chain, and whole
// sites per thread made four full waves and a nearly empty one on 20^3 x 40.
// Measured, us, with whole sites and so (2^4, 8^4, 16^4, 16^3 x 32, 20^3 x 40): 36
// 52 89 163 361 and 29 31 87 148 349 (the FP64 kernel 917 on the last).
// Bounds, for any matrices that pass the row test (not only unitary ones): rows of
// norm 1.025 give rows of X and Y of norm up to sqrt(3) 1.025^2 = 1.82, so a row's
// share of the trace is below 3.4 and is widened before the next one's (the trace
// itself may be 9.9, more than one accumulator holds).
template <typename T>
__global__ void __launch_bounds__(256, 2) k_plaquette_fx(const void* Uall, Geom g, int bpf,
                                                         double* __restrict__ partial) {
    typedef typename Vec2<T>::type V;
    const int f = blockIdx.x / (2 * bpf), half = threadIdx.x >> 7;
    const int s2 = (blockIdx.x - f * 2 * bpf) * 128 + (threadIdx.x & 127);  // 0 .. 2*vh-1
    const V* U = reinterpret_cast<const V*>(Uall) + (size_t)f * link_elems(g);
    const size_t vh = (size_t)g.vh;
    double slow = 0.0;
    long long acc = 0;  // units of 2^-57: at most 3 * 9.9
    if (s2 < 2 * g.vh) {
        const int p = s2 / g.vh, s = s2 - p * g.vh;
        int c[4];
        eo_coords(g, p, s, c);
#pragma unroll 1
        for (int mu = half; mu < 1 + 2 * half; ++mu) {
            const int smu = eo_neighbor(g, c, mu, +1);
#pragma unroll 1
            for (int nu = mu + 1; nu < 4; ++nu) {
                const V* ua = U + lidx(g, mu, p, 0, s);
                const V* ub = U + lidx(g, nu, p ^ 1, 0, smu);
                const V* uc = U + lidx(g, mu, p ^ 1, 0, eo_neighbor(g, c, nu, +1));
                const V* ud = U + lidx(g, nu, p, 0, s);
                cfx b[9], m[9];
                bool bad = fx_load_matrix(ub, 3 * vh, vh, b);
                bad = fx_load_matrix(uc, 3 * vh, vh, m) || bad;
                long long tr = 0;
#pragma unroll 1
                for (int i = 0; i < 3; ++i) {
                    cfx ra[3], rd[3], x[3], y[3];
                    float na = 0.f, nd = 0.f;
                    unsigned big = 0;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const V va = ua[(3 * i + k) * vh], vd = ud[(3 * i + k) * vh];
                        big = max(max(big, max(fx_magnitude(va.x), fx_magnitude(va.y))),
                                  max(fx_magnitude(vd.x), fx_magnitude(vd.y)));
                        ra[k].re = fx_of(va.x);
                        ra[k].im = fx_of(va.y);
                        rd[k].re = fx_of(vd.x);
                        rd[k].im = fx_of(vd.y);
                        na = fmaf((float)ra[k].re.h, (float)ra[k].re.h, fmaf((float)ra[k].im.h, (float)ra[k].im.h, na));
                        nd = fmaf((float)rd[k].re.h, (float)rd[k].re.h, fmaf((float)rd[k].im.h, (float)rd[k].im.h, nd));
                    }
                    bad = bad || big > kFxMagnitude || !(fabsf(na * 0x1p-56f - 1.f) < 0.05f) ||
                          !(fabsf(nd * 0x1p-56f - 1.f) < 0.05f);
                    m3fx_row<false>(ra, b, x);
                    m3fx_row<false>(rd, m, y);
                    facc t = facc_zero();
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        fx_mac(t, x[k].re, y[k].re);
                        fx_mac(t, x[k].im, y[k].im);
                    }
                    tr += facc_get(t) >> 3;
                }
                if (bad)
                    slow += plaquette_f64(ua, ub, uc, ud, vh);
                else
                    acc += tr;
            }
        }
    }
    __shared__ double red[8];
    const double tot = block_sum((fx_double(acc) * 8.0 + slow) / 3.0, red);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

}  // namespace

int launch_apply_gauge_fx(void* U, const void* G, const Geom& g, int nfields, cudaStream_t st) {
    k_apply_gauge_fx<false><<<blocks(8LL * g.vh * nfields, 128), 128, 0, st>>>((double2*)U, G, nullptr, nullptr, g,
                                                                                   nfields);
    MCG_CK(cudaGetLastError());
    note_launches(1);
    return 0;
}

int launch_handoff_fx(const void* W32, const void* W32lo, double* U64, double* G64, const Geom& g, int nfields,
                      cudaStream_t st) {
    int rc = 0;
    int4* Wfx = (int4*)scratch_device("handoff.W64", sizeof(int4) * gauge_elems(g) * nfields, &rc);
    if (rc) return rc;
    k_handoff_gauge_fx<<<blocks(2LL * g.vh * nfields, 128), 128, 0, st>>>(
        (const float4*)W32, (const float4*)W32lo, Wfx, (double2*)G64, g, nfields);
    k_apply_gauge_fx<true><<<blocks(8LL * g.vh * nfields, 128), 128, 0, st>>>(
        (double2*)U64, Wfx, (const float4*)W32, (const float4*)W32lo, g, nfields);
    MCG_CK(cudaGetLastError());
    note_launches(2);
    return 0;
}

void launch_plaquette_partials(const void* U, int prec, const Geom& g, int bpf, int nfields, double* partial,
                               cudaStream_t st) {
    const unsigned nb = 2u * (unsigned)bpf * nfields;
    if (prec == MCG_F64)
        k_plaquette_fx<double><<<nb, 256, 0, st>>>(U, g, bpf, partial);
    else
        k_plaquette_fx<float><<<nb, 256, 0, st>>>(U, g, bpf, partial);
}

// index-check counter of this unit (MCG_CHECK builds)
MCG_BOUND_READER(bound_hits_field_fx)

}  // namespace mcg
