// Wilson loops of FP64 SU(3) fields in fixed-point arithmetic (mcg_fx.cuh): line
// products S(x) = U(x) U(x + mu) ... in lexicographic site order as 64-bit
// integers (entry e of site x at L[e V + x]), and the loops closed from them.
#include <cuda_runtime.h>

#include "mcg_common.cuh"
#include "mcg_fx.cuh"
#include "mcg_internal.h"

namespace mcg {

namespace {

constexpr int WT = 128;

__device__ __forceinline__ void lex_coords(const Geom& g, int x, int c[4]) {
    c[0] = x % g.n[0];
    int r = x / g.n[0];
    c[1] = r % g.n[1];
    r /= g.n[1];
    c[2] = r % g.n[2];
    c[3] = r / g.n[2];
}
// lexicographic index of c + d, periodic, any signs; also its coordinates
__device__ __forceinline__ int lex_moved(const Geom& g, const int c[4], int4 d, int q[4]) {
    const int dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const int v = (c[mu] + dd[mu]) % g.n[mu];
        q[mu] = v < 0 ? v + g.n[mu] : v;
    }
    return q[0] + g.n[0] * (q[1] + g.n[1] * (q[2] + g.n[2] * q[3]));
}

// entry e of site x of line field `line` (T - 1 of the temporal ones, the path of
// the spatial ones), n of them
__device__ __forceinline__ size_t line_idx(int V, int n, int line, int e, int x) {
#ifdef MCG_CHECK
    if (mcg_bad((unsigned)line >= (unsigned)n || (unsigned)e >= 9u || (unsigned)x >= (unsigned)V)) return 0;
#endif
    return ((size_t)line * 9 + e) * V + x;
}

// One step of up to three paths at once (blockIdx.y): Pout(x) = Pin(x) times the
// link of direction `axis` at x + from, daggered for a backward step (from: the
// site the link starts at); first: Pin is the identity.
__global__ void __launch_bounds__(WT, 3) k_path_step_fx(const double2* __restrict__ U, const int4* __restrict__ Pin,
                                                        int4* __restrict__ Pout, Geom g, const PathSteps ps) {
    const int V = 2 * g.vh, x = blockIdx.x * WT + threadIdx.x;
    if (x >= V) return;
    const PathStep st = ps.step[blockIdx.y];
    const size_t off = line_idx(V, (int)gridDim.y, (int)blockIdx.y, 0, x);
    int c[4], q[4];
    lex_coords(g, x, c);
    const int y = lex_moved(g, c, make_int4(st.from[0], st.from[1], st.from[2], st.from[3]), q);
    const double2* u = U + lidx(g, st.axis, (q[0] + q[1] + q[2] + q[3]) & 1, 0, y >> 1);
    cfx a[9], b[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double2 v = u[(size_t)(st.back ? 3 * j + i : 3 * i + j) * g.vh];
            b[3 * i + j].re = fx_of(v.x);
            b[3 * i + j].im = fx_of(st.back ? -v.y : v.y);
        }
    if (ps.first) {
#pragma unroll
        for (int e = 0; e < 9; ++e) Pout[off + (size_t)e * V] = fx_pack(b[e]);
        return;
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) a[e] = fx_load(Pin + off + (size_t)e * V);
    m3fx_mul_inplace<false>(a, b);
#pragma unroll
    for (int e = 0; e < 9; ++e) Pout[off + (size_t)e * V] = fx_pack(a[e]);
}

// Per-block partials of the sum over sites of (1/3) Re tr of the loops
// P(x) S_t(x + r) (S_t(x) P(x + T t))^dag, path blockIdx.z (displacement r), T =
// blockIdx.y + 1, St the temporal lines of length 1 .. gridDim.y.  All T of a
// separation in one launch; X = P S_t and Y = S_t P row by row, sum Re X Y^*.
// Bound by the integer multiplier (two products per loop).  Measured on 12^3 x 24:
// 104 us for the 24 loops per site of one separation, where the FP64 kernel (one
// launch per T, FP64 pipe 91 %) took 900 us; lines of three axes in one launch
// fill a lattice that one axis leaves at two warps per scheduler.
__global__ void __launch_bounds__(WT, 4) k_wilson_fx(const int4* __restrict__ P, const int4* __restrict__ St, Geom g,
                                                     const PathSteps ps, double* __restrict__ partial) {
    const int V = 2 * g.vh, x = blockIdx.x * WT + threadIdx.x;
    const size_t sV = (size_t)V;
    long long sum = 0;
    if (x < V) {
        const PathStep st = ps.step[blockIdx.z];
        const int4* Pz = P + line_idx(V, (int)gridDim.z, (int)blockIdx.z, 0, 0);
        const int4* L = St + line_idx(V, (int)gridDim.y, (int)blockIdx.y, 0, 0);
        int c[4], q[4];
        lex_coords(g, x, c);
        const int xr = lex_moved(g, c, make_int4(st.from[0], st.from[1], st.from[2], st.from[3]), q);
        const int xt = lex_moved(g, c, make_int4(0, 0, 0, (int)blockIdx.y + 1), q);
        cfx a[9], b[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            a[e] = fx_load(L + line_idx(V, 1, 0, e, xr));
            b[e] = fx_load(Pz + line_idx(V, 1, 0, e, xt));
        }
        facc t = facc_zero();
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {
            cfx rp[3], rs[3], X[3], Y[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                rp[k] = fx_load(Pz + (3 * i + k) * sV + x);
                rs[k] = fx_load(L + (3 * i + k) * sV + x);
            }
            m3fx_row<false>(rp, a, X);
            m3fx_row<false>(rs, b, Y);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                fx_mac(t, X[k].re, Y[k].re);
                fx_mac(t, X[k].im, Y[k].im);
            }
        }
        sum = (facc_get(t) + 64) >> 7;  // units of 2^-53, at most 3.1
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    __shared__ double red[WT / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = fx_double(sum) * 128.0;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < WT / 32; ++k) s += red[k];
        partial[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s / 3.0;
    }
}

// out[y out_stride] = scale times the sum of the partials of T = y + 1 over npath
// paths, in a fixed order
__global__ void __launch_bounds__(256) k_sum_loops(const double* __restrict__ partial, int nb, int npath, double scale,
                                                   double* __restrict__ out) {
    double v = 0.0;
    for (int z = 0; z < npath; ++z)
        for (int k = threadIdx.x; k < nb; k += blockDim.x)
            v += partial[((size_t)z * gridDim.x + blockIdx.x) * nb + k];
    __shared__ double red[8];
    const double tot = block_sum(v, red);
    if (threadIdx.x == 0) out[blockIdx.x] = tot * scale;
}

}  // namespace

int wilson_fx_blocks(const Geom& g) { return (2 * g.vh + WT - 1) / WT; }

void launch_path_step_fx(const double* U, const void* Pin, void* Pout, const Geom& g, const PathSteps& ps, int npath,
                         cudaStream_t st) {
    k_path_step_fx<<<dim3(wilson_fx_blocks(g), npath), WT, 0, st>>>((const double2*)U, (const int4*)Pin, (int4*)Pout, g,
                                                                    ps);
}

void launch_wilson_fx(const void* P, const void* St, const Geom& g, const PathSteps& ps, int npath, int Tmax,
                      double* partial, double scale, double* out, cudaStream_t st) {
    const int nb = wilson_fx_blocks(g);
    k_wilson_fx<<<dim3(nb, Tmax, npath), WT, 0, st>>>((const int4*)P, (const int4*)St, g, ps, partial);
    k_sum_loops<<<Tmax, 256, 0, st>>>(partial, nb, npath, scale, out);
}

// index-check counter of this unit (MCG_CHECK builds)
MCG_BOUND_READER(bound_hits_wilson_fx)

}  // namespace mcg
