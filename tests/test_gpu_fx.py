"""FP64 paths in fixed-point arithmetic (mcg_fx.cuh) against the FP64 oracle
at the edges of their ranges: lattices of extent 2 (a neighbour reached from
both sides), ragged tails of the blocks, several fields per call, staple
weights up to the limit of the fixed-point step and just above it (the FP64
kernels)."""
import numpy as np
import pytest

import oracle
from paper_0807_0264_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _pack(mcg, Us, dims):
    return mcg.mcg_pack_links(torch.from_numpy(np.ascontiguousarray(np.stack(Us))).cuda(), dims)


# rho (6 |cp| + 18 |cr|) at, below and above the limit 1; n even and odd (the
# two buffers); the oracle rounds ~150 times per link and step at 1.1e-16
# relative to entries of at most 1: 2e-14 per step
@pytest.mark.parametrize("rho,eps,n", [(1 / 6, 1.0, 3), (0.1667, 1.0, 2), (0.07751937984496124, -0.25, 2),
                                       (-0.1, 1.0, 1), (0.06, -0.25, 5), (1e-9, 1.0, 2), (0.0, 0.5, 1)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 10, 4), (4, 14, 2, 6)])
def test_fixed_point_smear(dims, rho, eps, n):
    from paper_0807_0264_gb300 import mcg

    Us = [synth.make_field(dims, w, s) for w, s in ((0.5, 1), (3.0, 2), (0.0, 3))]
    S = mcg.mcg_unpack_links(mcg.mcg_smear(_pack(mcg, Us, dims), dims, rho, eps, n), dims).cpu().numpy()
    for U, s in zip(Us, S):
        assert np.abs(s - oracle.smear(dims, U, rho, eps, n)).max() < 2e-14 * n


# lattices of the three shapes of the half-sweep (8, 4 and 2 threads per site), with and without a ragged last
# block; a field near its maximum, whose local problems are well conditioned: the FP64 sweep's bar of 1e-11 per
# link; nfields = 2 runs them as chains
@pytest.mark.parametrize("dims,nf", [((2, 2, 2, 2), 1), ((6, 2, 10, 14), 2), ((10, 6, 14, 12), 1), ((14, 14, 14, 14), 1)])
def test_fixed_point_sweep(dims, nf):
    from paper_0807_0264_gb300 import mcg

    Us = [synth.make_field(dims, 0.4, s, gauge=False) for s in range(nf)]
    Ud, Gd = _pack(mcg, Us, dims), mcg.identity_gauge(dims, nf)
    r = mcg.mcg_fix(Ud, Gd, dims, mcg.Params(tol=-1e300, max_sweeps=2, reunit_every=0))
    Uo, Go = mcg.mcg_unpack_links(Ud, dims).cpu().numpy(), mcg.mcg_unpack_gauge(Gd, dims).cpu().numpy()
    for f, U in enumerate(Us):
        ref = oracle.fix(dims, U, tol=-1e300, max_sweeps=2, reunit_every=0)
        assert np.abs(Uo[f] - ref["U"]).max() < 1e-11 and np.abs(Go[f] - ref["G"]).max() < 1e-11
        assert abs(r["R"][f] - ref["R_hist"][-1]) < 1e-12 * ref["R_hist"][-1]


# rough fields from random transforms: most local problems leave the warm start (the second seed, the Jacobi seed
# and the FP64 solve all run).  A problem with relative gap g between the multiplier and lambda_max moves its
# element by ~1e-15 / g and P(gap < g) ~ g, so one link in a thousand may pass 1e-12 tenfold: the bar on the
# 99.9 % quantile; R is stationary in each element
@pytest.mark.parametrize("seed", range(4))
def test_fixed_point_sweep_rough(seed):
    from paper_0807_0264_gb300 import mcg

    dims = (6, 4, 6, 8)
    U, G = synth.make_field(dims, 3.0, seed), synth.random_gauge(dims, 50 + seed)
    Ud, Gd = _pack(mcg, [U], dims), mcg.mcg_pack_gauge(torch.from_numpy(G).unsqueeze(0).cuda(), dims)
    r = mcg.mcg_fix(Ud, Gd, dims, mcg.Params(tol=-1e300, max_sweeps=1, reunit_every=0))
    ref = oracle.fix(dims, U, G, tol=-1e300, max_sweeps=1, reunit_every=0)
    err = np.abs(mcg.mcg_unpack_links(Ud, dims)[0].cpu().numpy() - ref["U"])
    assert np.quantile(err, 0.999) < 1e-11
    assert abs(r["R"][0] - ref["R_hist"][-1]) < 1e-11 * ref["R_hist"][-1]


def test_unvalidated_sites_keep_the_fp64_kernel():
    """mcg_halfsweep_slab takes any matrices: sites next to a link outside the fixed-point range (scaled by 3 and
    by 1/4, zero) agree with the oracle as all others do (F scales with the square of the
    links: 9 x the 1e-11 bar)."""
    from paper_0807_0264_gb300 import mcg

    dims = (4, 6, 2, 6)
    U, G = synth.make_field(dims, 0.4, 5, gauge=False), synth.identity_gauge(dims)
    U[7, 2] *= 3.0
    U[20, 0] *= 0.25
    U[100, 3] = 0.0
    Ud, Gd = _pack(mcg, [U], dims), mcg.mcg_pack_gauge(torch.from_numpy(G).unsqueeze(0).cuda(), dims)
    Uo, Go = U.copy(), G.copy()
    for parity in (0, 1):
        R = mcg.mcg_halfsweep_slab(Ud, Gd, dims, parity, 0, dims[3], want_R=parity == 1)
        oracle.halfsweep_slab(dims, Uo, Go, parity, 0, dims[3])
    assert np.abs(mcg.mcg_unpack_links(Ud, dims)[0].cpu().numpy() - Uo).max() < 9e-11
    assert np.abs(mcg.mcg_unpack_gauge(Gd, dims)[0].cpu().numpy() - Go).max() < 9e-11
    ref = (np.abs(np.trace(Uo, axis1=-2, axis2=-1)) ** 2).sum()
    assert abs(R - ref) < 1e-11 * ref


# near-unitary fields take the fixed-point kernels, the others (one field scaled, one with a zero and a scaled
# link) FP64 per link or plaquette; FP32 fields are exact inputs of both.  Rounding: ~30 operations of 1.1e-16 on
# entries of the size of a plaquette's factors (a transformed link), averaged over the plaquettes
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 10, 4), (10, 6, 14, 12)])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 7.0, None])
def test_fixed_point_plaquette_and_transforms(dims, scale):
    from paper_0807_0264_gb300 import mcg

    U = synth.make_field(dims, 0.7, 8)
    if scale is None:
        U[3, 1] *= 40.0
        U[9, 2] = 0.0
    else:
        U *= scale
    Ud = _pack(mcg, [U, U], dims)
    ref, top = oracle.plaquette(dims, U), max(1.0, np.abs(U).max()) ** 4 if scale is None else scale**4
    assert np.abs(np.array(mcg.mcg_plaquette(Ud, dims)) - ref).max() < 1e-14 * top
    U32 = mcg.mcg_convert(Ud, mcg.F32)
    ref32 = oracle.plaquette(dims, mcg.mcg_unpack_links(U32, dims)[0].cpu().numpy())
    assert np.abs(np.array(mcg.mcg_plaquette(U32, dims)) - ref32).max() < 1e-14 * top
    # an ascent step: W = exp(i alpha grad.lambda / 2) on the links and on Omega
    G = mcg.identity_gauge(dims, 2)
    grad = torch.randn(2, np.prod(dims), 8, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    mcg.mcg_ascent_step(Ud, G, grad, dims, 0.1)
    W = mcg.mcg_unpack_gauge(G, dims).cpu().numpy()
    got = mcg.mcg_unpack_links(Ud, dims).cpu().numpy()
    for f in range(2):
        assert np.abs(got[f] - oracle.apply_gauge(dims, U, W[f])).max() < 1e-14 * max(1.0, np.abs(U).max())


# the reverse step: lattices of extent 2 (a link in its own staples), gradients of any scale, zero but for one
# link, and with infinities; links that are not near-unitary take the FP64 kernel.  The oracle's bar of the FP64
# kernel (1e-11 of the gradient), for a gradient of one link relative to what it reaches
@pytest.mark.parametrize("eps,rho", [(1.0, 0.1), (-0.25, 0.06), (1.0, 0.3)])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 2), (4, 4, 2, 6)])
def test_fixed_point_smear_backward(dims, eps, rho):
    from paper_0807_0264_gb300 import mcg

    rng = np.random.default_rng(4)
    U, V = synth.make_field(dims, 0.7, 9), np.prod(dims)
    dense = rng.standard_normal((V, 4, 3, 3)) + 1j * rng.standard_normal((V, 4, 3, 3))
    point = np.zeros_like(dense)
    point[V // 3, 1] = dense[V // 3, 1]

    def step(U, G):
        return mcg.mcg_unpack_links(mcg.mcg_smear_backward_step(_pack(mcg, [U], dims), _pack(mcg, [G], dims), dims, rho, eps),
                                    dims)[0].cpu().numpy()

    for G in (dense, point):  # the step is linear: scales by powers of ten against the scaled reference
        ref = oracle.smear_step_backward(dims, U, G, rho, eps)
        for scale in (1.0, 1e-200, 1e150):
            assert np.abs(step(U, scale * G) / scale - ref).max() < 1e-11 * np.abs(ref).max()
    assert not step(U, np.zeros_like(dense)).any()
    Ub = U.copy()
    Ub[0, 0] *= 1.5
    ref = oracle.smear_step_backward(dims, Ub, dense, rho, eps)
    assert np.abs(step(Ub, dense) - ref).max() < 1e-11 * np.abs(ref).max()
    bad = dense.copy()
    bad[1, 2, 0, 0] = np.inf
    assert not np.isfinite(step(U, bad)).all()


# loops of SU(3) fields (fixed point) and of others (FP64): long lines, every T of a separation in one launch, odd
# remainders of the 128-site blocks; ~L roundings of 1.1e-16 on a line of L links, bar 1e-15 L
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 10, 6), (4, 4, 4, 14)])
@pytest.mark.parametrize("scale", [1.0, 1.001])
def test_fixed_point_wilson_loops(dims, scale):
    from paper_0807_0264_gb300 import mcg

    R, T = min(dims[:3]), dims[3]
    U = [scale * synth.make_field(dims, 0.3, s, gauge=s == 1) for s in (1, 2)]
    W = mcg.mcg_wilson_loops(_pack(mcg, U, dims), dims, R, T)
    vec = [(1, 0, 0), (1, 1, 0)] if R == 2 else [(1, 2, 1), (0, 1, 3), (2, 2, 0)]
    Wo = mcg.mcg_wilson_loops_offaxis(_pack(mcg, U, dims), dims, vec, T)
    for f in range(2):
        top = scale ** (2 * (R + T + 3))
        assert np.abs(W[f] - oracle.wilson_loops(dims, U[f], R, T)).max() < 1e-15 * (2 * (R + T)) * top
        assert np.abs(Wo[f] - oracle.wilson_loops_offaxis(dims, U[f], vec, T)).max() < 1e-15 * (2 * (4 + T)) * top


def test_observables_at_their_edges():
    """The FP32 filter of the center projection and the exact halvings of the vortex removal against the oracle, bit
    for bit: traces on and next to
    the sector boundaries, zeros of both signs, subnormal and huge entries, infinities."""
    from paper_0807_0264_gb300 import mcg

    dims, rng = (4, 4, 2, 6), np.random.default_rng(6)
    V = int(np.prod(dims))
    U = (rng.standard_normal((V, 4, 3, 3)) + 1j * rng.standard_normal((V, 4, 3, 3))) * 10.0 ** rng.integers(-9, 3, (V, 4, 1, 1))
    t = np.array([1.0, np.sqrt(3.0), np.nextafter(np.sqrt(3.0), 2), np.nextafter(np.sqrt(3.0), 1), 0.0, 1e-5, 9e-6, 1e-300])
    for k in range(V):  # traces x + i y near the rays |y| = sqrt(3) x and y = 0, split unevenly over the diagonal
        x, y = rng.choice(t) * rng.choice([1, -1]), rng.choice(t) * rng.choice([1, -1])
        U[k, 1] = 0.0
        U[k, 1, 0, 0], U[k, 1, 1, 1], U[k, 1, 2, 2] = (x + 1j * y) - 0.25, 0.5, -0.25
    U[0, 2, 0, 1], U[1, 2, 0, 1], U[2, 2, 0, 1] = 5e-324, 1e308 + 1j * 1e308, -0.0
    U[3, 2, 1, 1] = 2.3e-308 - 1j * 4.4e-308
    Ud = _pack(mcg, [U], dims)
    Z, _ = mcg.mcg_center_project(Ud, dims)
    m = mcg.mcg_unpack_center(Z, dims)[0].cpu().numpy()
    assert np.array_equal(m, oracle.center_project(dims, U))
    Ur, _ = mcg.mcg_vortex_remove(Ud, Z, dims)
    assert np.array_equal(mcg.mcg_unpack_links(Ur, dims)[0].cpu().numpy(), oracle.vortex_remove(dims, U, m))
    W = np.where(np.abs(U) > 1e100, 0, U)
    for scale in (1.0, 1e-3, 0.02):  # ~10 roundings of 1.1e-16
        R = mcg.mcg_functional(_pack(mcg, [scale * W], dims), dims)[0]
        ref = (np.abs(np.trace(scale * W, axis1=-2, axis2=-1)) ** 2).sum()
        assert abs(R - ref) < 2e-15 * ref
    S = synth.make_field(dims, 0.4, 2)
    assert abs(mcg.mcg_functional(_pack(mcg, [S], dims), dims)[0] - oracle.functional_R(dims, S)) < 2e-15 * oracle.functional_R(dims, S)
    for entry in (np.inf, -np.inf, np.nan):  # refused as before, wherever it stands
        B = S.copy()
        B[V - 1, 3, 2, 2] = entry
        for call in (lambda: mcg.mcg_center_project(_pack(mcg, [B], dims), dims), lambda: mcg.mcg_smear(_pack(mcg, [B], dims), dims, 0.1, 1.0, 1)):
            with pytest.raises(mcg.MCGError):
                call()
    for off, ok in ((5e-7, True), (2e-6, False)):  # the SU(3) tolerance of 1e-6
        B = S.copy()
        B[1, 1] *= 1 + off / 3
        if ok:
            mcg.mcg_smear(_pack(mcg, [B], dims), dims, 0.1, 1.0, 1)
        else:
            with pytest.raises(mcg.MCGError):
                mcg.mcg_smear(_pack(mcg, [B], dims), dims, 0.1, 1.0, 1)


# kept sweep graphs: calls alternating between shapes, schedules, precisions and batch sizes (more of them than are
# kept), with other fields and other streams, before and after mcg_release, return the bits of their first call
def test_repeated_fixes_with_kept_graphs():
    from paper_0807_0264_gb300 import mcg

    P = mcg.Params
    kinds = [(4, P(tol=1e-9, max_sweeps=90, check_every=5)), (4, P(tol=1e-9, max_sweeps=90, check_every=7)),
             (4, P(tol=1e-4, max_sweeps=90, check_every=5)), (4, P(tol=1e-9, max_sweeps=90, reunit_every=3)),
             (6, P(tol=1e-9, max_sweeps=40)), (4, P(tol=1e-9, max_sweeps=90, fp32_sweeps=60)),
             (4, P(tol=1e-9, max_sweeps=90, fp32_sweeps=60, fp64_df=1)), (4, P(tol=1e-9, max_sweeps=90, fp64_solve32=1))]
    data = {(n, s): (synth.make_field((n, 4, 4, 6), 2.0, s)) for n in (4, 6) for s in range(3)}

    def run(kind, seeds, stream):
        n, prm = kinds[kind]
        dims = (n, 4, 4, 6)
        with torch.cuda.stream(stream):
            Us = [_pack(mcg, [data[n, s]], dims) for s in seeds]
            Gs = [mcg.identity_gauge(dims) for _ in seeds]
            r = mcg.mcg_fix_batch(Us, Gs, [dims] * len(Us), prm)
            return r["R"], r["sweeps"], [u.cpu().numpy().tobytes() for u in Us + Gs]

    main, side = torch.cuda.current_stream(), torch.cuda.Stream()
    calls = [(k, seeds) for k in range(len(kinds)) for seeds in ((0,), (1, 2), (1,))]
    first = {c: run(*c, main) for c in calls}
    for c in calls[::-1]:
        assert run(*c, side) == first[c]
    mcg.mcg_release()
    for c in calls[::2]:
        assert run(*c, main) == first[c]


# the input check of a batch in one launch per 32 arrays: the message is that of the first bad array in the order
# U_0, G_0, U_1, ..., wherever its blocks lie, and no field is touched
@pytest.mark.parametrize("prec", ["F64", "F32"])
@pytest.mark.parametrize("bad,which", [(0, "U"), (15, "G"), (16, "U"), (19, "G")])
def test_batched_input_check(prec, bad, which):
    from paper_0807_0264_gb300 import mcg

    prec = getattr(mcg, prec)
    dl = [(2, 2, 2, 2), (6, 2, 10, 4), (4, 14, 2, 6)] * 6 + [(8, 8, 4, 4), (2, 4, 2, 2)]
    Us = [mcg.mcg_pack_links(torch.from_numpy(synth.make_field(d, 1.0, i)).unsqueeze(0).cuda(), d, prec)
          for i, d in enumerate(dl)]
    Gs = [mcg.identity_gauge(d, 1, prec) for d in dl]
    (Us if which == "U" else Gs)[bad].view(-1)[-1] += 0.5
    Us[19].view(-1)[0] = float("nan")
    before = [x.clone() for x in Us + Gs]
    name = which if bad < 19 else "U"
    with pytest.raises(RuntimeError, match=f"mcg_fix_batch: {name}: 1 matrices are not finite"):
        mcg.mcg_fix_batch(Us, Gs, dl, mcg.Params(max_sweeps=2))
    for x, y in zip(Us + Gs, before):
        assert torch.equal(torch.nan_to_num(x, nan=9.0), torch.nan_to_num(y, nan=9.0))


# calls enqueued on several streams without a wait between them share the smearing scratch: each returns the bits of
# its own call made alone.  In a captured graph (with no scratch allocated) the backward step runs the FP64 kernel:
# both round ~300 times per link relative to the gradient's size, 1e-13
def test_smear_calls_on_several_streams_and_captured():
    from paper_0807_0264_gb300 import mcg

    dims, gen = (8, 8, 8, 16), torch.Generator(device="cuda").manual_seed(5)
    Us = [_pack(mcg, [synth.make_field(dims, 1.0, s)], dims) for s in range(4)]
    Gs = [torch.randn(U.shape, dtype=U.dtype, device="cuda", generator=gen) for U in Us]
    for eps, rho in ((1.0, 0.1), (-0.25, 0.06)):
        alone = []
        for U, G in zip(Us, Gs):
            alone.append((mcg.mcg_smear(U, dims, rho, eps, 1), mcg.mcg_smear_backward_step(U, G, dims, rho, eps)))
            torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in Us]
        outs = [[] for _ in Us]
        for _ in range(3):
            for st, U, G, o in zip(streams, Us, Gs, outs):
                with torch.cuda.stream(st):
                    o.append((mcg.mcg_smear(U, dims, rho, eps, 1), mcg.mcg_smear_backward_step(U, G, dims, rho, eps)))
        torch.cuda.synchronize()
        for o, (s, b) in zip(outs, alone):
            assert all(torch.equal(x, s) and torch.equal(y, b) for x, y in o)
        mcg.mcg_release()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = mcg.mcg_smear_backward_step(Us[0], Gs[0], dims, rho, eps)
        graph.replay()
        torch.cuda.synchronize()
        assert float((out - alone[0][1]).abs().max()) < 1e-13 * float(alone[0][1].abs().max())


# re-unitarisation in the kernel that ends the sweep: after every sweep, every third, and only past the last one; fields
# of several sizes as chains and in one launch; the sweep test's bar of 1e-11 per link for fields near a maximum
@pytest.mark.parametrize("every", [1, 3, 4])
@pytest.mark.parametrize("copies", [1, 6])
def test_reunitarise_at_the_end_of_a_sweep(every, copies):
    from paper_0807_0264_gb300 import mcg

    dl = [(2, 2, 2, 2), (4, 6, 2, 4), (6, 2, 10, 14)]
    Uh = [synth.make_field(d, 0.4, i, gauge=False) for i, d in enumerate(dl)]
    Us = [_pack(mcg, [U], d) for _ in range(copies) for U, d in zip(Uh, dl)]
    Gs = [mcg.identity_gauge(d) for _ in range(copies) for d in dl]
    mcg.mcg_fix_batch(Us, Gs, dl * copies, mcg.Params(tol=-1e300, max_sweeps=3, reunit_every=every, check_every=2))
    refs = [oracle.fix(d, U, tol=-1e300, max_sweeps=3, reunit_every=every) for U, d in zip(Uh, dl)]
    for k, (U, G) in enumerate(zip(Us, Gs)):
        d, ref = dl[k % 3], refs[k % 3]
        assert np.abs(mcg.mcg_unpack_links(U, d)[0].cpu().numpy() - ref["U"]).max() < 1e-11
        assert np.abs(mcg.mcg_unpack_gauge(G, d)[0].cpu().numpy() - ref["G"]).max() < 1e-11
