"""FP64 entry points at the limits of their fixed-point kernels: links that are not unitary though their rows are
of unit norm, schedules and batches."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_0807_0264_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _pack(mcg, Us, dims):
    return mcg.mcg_pack_links(torch.from_numpy(np.ascontiguousarray(np.stack(Us))).cuda(), dims)


def _unit_rows(dims, diagonal, scale=1.0):
    """Every link the all-ones matrix plus `diagonal` times the identity, its rows normalised to `scale`."""
    m = np.ones((3, 3)) + diagonal * np.eye(3)
    m *= scale / np.linalg.norm(m[0])
    return np.broadcast_to(m.astype(complex), (int(np.prod(dims)), 4, 3, 3)).copy()


# rows of norm 1 that are not orthogonal: a plaquette of 9, beyond the 8 that one sum of the fixed point holds (row norms
# to 1.02 pass the kernel's test; the last case fills the low halves too).  ~30 roundings of 1.1e-16 relative to 9 / 3
@pytest.mark.parametrize("diagonal,scale", [(0.0, 1.0), (0.1, 1.0), (0.2, 1.0), (-0.5, 1.0), (0.0, 1.02), (0.0, 1.0199999)])
def test_plaquette_of_rows_that_are_not_orthogonal(diagonal, scale):
    from paper_0807_0264_gb300 import mcg

    dims = (4, 2, 6, 4)
    U = _unit_rows(dims, diagonal, scale)
    ref = oracle.plaquette(dims, U)
    Ud = _pack(mcg, [U, U], dims)
    out = torch.empty(2, dtype=torch.float64, device="cuda")
    assert np.abs(np.array(mcg.mcg_plaquette(Ud, dims)) - ref).max() < 2e-14
    assert np.abs(mcg.mcg_plaquette_static(Ud, dims, out).cpu().numpy() - ref).max() < 2e-14
    U32 = mcg.mcg_convert(Ud, mcg.F32)
    ref32 = oracle.plaquette(dims, mcg.mcg_unpack_links(U32, dims)[0].cpu().numpy())
    assert np.abs(np.array(mcg.mcg_plaquette(U32, dims)) - ref32).max() < 2e-14


# the reverse step of such links (staple sums of 10 before the weight), and of links just inside the test (None: inner
# products of rows below 0.01, squared row norms 1.014): the bar of the FP64 kernel, 1e-11 of the gradient
@pytest.mark.parametrize("diagonal", [0.0, 0.1, 1.0, None])
@pytest.mark.parametrize("eps,rho", [(1.0, 1 / 6), (-0.25, 0.06)])
def test_smear_backward_of_rows_that_are_not_orthogonal(diagonal, eps, rho):
    from paper_0807_0264_gb300 import mcg

    dims, rng = (4, 2, 6, 4), np.random.default_rng(3)
    if diagonal is None:
        U = synth.make_field(dims, 0.7, 3)
        U[..., 0, :] += 0.009 * U[..., 1, :]
        U *= 1.007 / np.linalg.norm(U, axis=-1, keepdims=True)
    else:
        U = _unit_rows(dims, diagonal)
    G = rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape)
    got = mcg.mcg_smear_backward_step(_pack(mcg, [U], dims), _pack(mcg, [G], dims), dims, rho, eps)
    ref = oracle.smear_step_backward(dims, U, G, rho, eps)
    assert np.abs(mcg.mcg_unpack_links(got, dims)[0].cpu().numpy() - ref).max() < 1e-11 * np.abs(ref).max()


# a half-sweep of links a few percent or less off unitarity, with one link far off: a site moves once, whatever the
# norms of its rows after the move, and counts once in R.  The FP64 sweep's bar of 1e-11 per link near a maximum,
# 9 times that for the link scaled by 3
@pytest.mark.parametrize("overlap,scale", [(0.1, 1.0), (0.1, 1.02), (0.009, 1.007), (0.007, 0.994)])
def test_halfsweep_of_links_off_unitarity(overlap, scale):
    from paper_0807_0264_gb300 import mcg

    dims = (4, 6, 4, 6)
    U, G = synth.make_field(dims, 0.4, 5, gauge=False), synth.identity_gauge(dims)
    U[..., 0, :] += overlap * U[..., 1, :]
    U *= scale / np.linalg.norm(U, axis=-1, keepdims=True)
    U[7, 2] *= 3.0
    Ud, Gd = _pack(mcg, [U], dims), mcg.mcg_pack_gauge(torch.from_numpy(G).unsqueeze(0).cuda(), dims)
    Uo, Go = U.copy(), G.copy()
    for sweep in range(2):
        for parity in (0, 1):
            R = mcg.mcg_halfsweep_slab(Ud, Gd, dims, parity, 0, dims[3], want_R=parity == 1)
            oracle.halfsweep_slab(dims, Uo, Go, parity, 0, dims[3])
    assert np.abs(mcg.mcg_unpack_links(Ud, dims)[0].cpu().numpy() - Uo).max() < 9e-11
    assert np.abs(mcg.mcg_unpack_gauge(Gd, dims)[0].cpu().numpy() - Go).max() < 9e-11
    ref = (np.abs(np.trace(Uo, axis1=-2, axis2=-1)) ** 2).sum()
    assert abs(R - ref) < 1e-11 * ref


# a preconditioned fix that ends at its sweep cap fills its results whether or not the caller asks for the sectors
def test_results_of_a_fix_at_its_cap_without_sectors():
    from paper_0807_0264_gb300 import mcg

    dims, prm = (4, 2, 6, 4), mcg.Params(tol=1e-12, max_sweeps=3)
    U = _pack(mcg, [synth.make_field(dims, 1.5, 4)], dims)
    Z = torch.empty((1, 4, 2, int(np.prod(dims)) // 2), dtype=torch.int8, device="cuda")
    runs = [mcg.mcg_precondition_fix(U.clone(), mcg.identity_gauge(dims), dims, prm, nsmear=2, Z=z)[0] for z in (Z, None)]
    assert runs[0] == runs[1] and runs[0]["status"] == 1 and runs[0]["sweeps_fixed"] == 3 and runs[0]["V_fixed"] > 0
    res = (mcg.mcg_precond_result * 1)()
    cp, ns, out, G = prm.c(), (mcg.ctypes.c_int * 1)(2), torch.empty_like(U), mcg.identity_gauge(dims)
    rc = mcg.library().mcg_precondition_levels(U.data_ptr(), out.data_ptr(), G.data_ptr(), None, mcg.lattice(dims, 1, mcg.F64),
                                               mcg.ctypes.byref(cp), 0.1, 1.0, ns, 1, mcg.F64, res, None)
    assert rc == 1 and res[0].as_dict() == runs[0]


# a level without smearing beside smeared ones, on schedules that keep some fields in FP64 arithmetic and not others:
# the bits of the level alone
@pytest.mark.parametrize("schedule", [dict(fp32_sweeps=60), dict(fp32_sweeps=60, fp64_df=1),
                                      dict(fp32_sweeps=60, fp64_solve32=1), dict()])
def test_unsmeared_level_beside_smeared_ones(schedule):
    from paper_0807_0264_gb300 import mcg

    dims = (6, 4, 4, 6)
    prm = mcg.Params(tol=1e-9, max_sweeps=120, check_every=10, **schedule)
    U = _pack(mcg, [synth.make_field(dims, 2.0, 4)], dims)
    Ua, Ga, _, ra = mcg.mcg_precondition_levels(U, dims, [0], prm)
    Ub, Gb, _, rb = mcg.mcg_precondition_levels(U, dims, [0, 2, 5], prm)
    Uc, Gc = U.clone(), mcg.identity_gauge(dims)
    rc = mcg.mcg_precondition_fix(Uc, Gc, dims, prm)
    for Ux, Gx, rx in ((Ub, Gb, rb), (Uc, Gc, rc)):
        assert torch.equal(Ux[:1], Ua) and torch.equal(Gx[:1], Ga)
        assert rx[0]["V_fixed"] == ra[0]["V_fixed"] and rx[0]["sweeps_fixed"] == ra[0]["sweeps_fixed"]


# plain FP64 sweeps: links, transform, R of every sweep and the stop sweep are those of the field alone, in batches for
# which the sweep takes 8, 4 and 2 threads per site, as chains and in one launch
@pytest.mark.parametrize("copies", [2, 4, 10, 17])
def test_fp64_batch_equals_the_field_alone(copies):
    from paper_0807_0264_gb300 import mcg

    dims = (8, 6, 10, 8)
    prm = mcg.Params(tol=1e-5, max_sweeps=25, reunit_every=10, check_every=5)
    fields = [synth.make_field(dims, 1.5, s) for s in (1, 2)]
    alone = []
    for U in fields:
        Ud, Gd = _pack(mcg, [U], dims), mcg.identity_gauge(dims)
        r = mcg.mcg_fix(Ud, Gd, dims, prm, history=True)
        alone.append((Ud, Gd, r["R"][0], r["sweeps"][0], np.asarray(r["R_hist"]).reshape(-1)))
    Ud, Gd = _pack(mcg, [fields[k % 2] for k in range(copies)], dims), mcg.identity_gauge(dims, copies)
    r = mcg.mcg_fix(Ud, Gd, dims, prm, history=True)
    hist = np.asarray(r["R_hist"]).reshape(copies, -1)
    for k in range(copies):
        U1, G1, R1, s1, h1 = alone[k % 2]
        assert r["sweeps"][k] == s1 and r["R"][k] == R1 and np.array_equal(hist[k], h1)
        assert torch.equal(Ud[k], U1[0]) and torch.equal(Gd[k], G1[0])


def test_time_halfsweep_follows_the_block_setting():
    """The FP64 timing, which the block size is tuned with, is of one launch of the kernel that reads the setting."""
    from paper_0807_0264_gb300 import mcg

    dims = (4, 4, 4, 6)
    U, G = _pack(mcg, [synth.make_field(dims, 0.4, 3)], dims), mcg.identity_gauge(dims)
    old = mcg.mcg_get_sweep_block(mcg.F64)
    try:
        for nt in (64, 128):
            mcg.mcg_set_sweep_block(mcg.F64, nt)
            n0 = mcg.mcg_kernel_launches()
            assert mcg.mcg_time_halfsweep(U, G, dims, 1, 5, False) > 0
            assert mcg.mcg_kernel_launches() - n0 == 5
        plain = mcg.autotune_schedule([U], [dims], mcg.Params(), trial_sweeps=4, chunks=(2, 4))
        assert plain["block"] == 128 and plain["precision"] == "f64"
        assert set(plain["ms_per_sweep"]) == {f"{b}x{c}" for b in (64, 128) for c in (2, 4)}
        s32 = mcg.autotune_schedule([U], [dims], mcg.Params(fp64_solve32=1), trial_sweeps=4, chunks=(2,))
        assert s32["block"] in (64, 128) and len(set(s32["ms_per_sweep"].values())) == 2
    finally:
        mcg.mcg_set_sweep_block(mcg.F64, old)


# the hand-off of a transform W that is not near-unitary at some sites, or not finite: the FP64 form there, as in the
# FP64 hand-off (~60 roundings of 1.1e-16; the links' transforms are unitary, entries at most 1)
@pytest.mark.parametrize("lo", [False, True])
def test_handoff_of_transforms_off_unitarity(lo):
    from paper_0807_0264_gb300 import mcg

    class Geom(ctypes.Structure):
        _fields_ = [("n", ctypes.c_int * 4), ("vh", ctypes.c_int)]

    fn = mcg.library()["_ZN3mcg14launch_handoffEPKvS1_PdS2_RKNS_4GeomEibP11CUstream_st"]
    fn.argtypes = [ctypes.c_void_p] * 4 + [ctypes.POINTER(Geom), ctypes.c_int, ctypes.c_bool, ctypes.c_void_p]
    dims = (4, 2, 6, 4)
    vh = int(np.prod(dims)) // 2
    g = Geom((ctypes.c_int * 4)(*dims), vh)
    W = synth.random_gauge(dims, 5)[:, :2].reshape(2 * vh, 6).astype(np.complex64)
    W[3] *= 1.5
    W[11, 2] = np.nan
    W[vh + 5, 4] += 0.3
    W[vh + 9] *= np.complex64(1e20)
    # compact storage: three chunks of two entries per matrix, (parity, chunk, site)
    chunks = np.ascontiguousarray(W.view(np.float32).reshape(2, vh, 3, 4).transpose(0, 2, 1, 3))
    Wd = torch.from_numpy(chunks).cuda()
    Wl = torch.from_numpy(1e-9 * np.random.default_rng(1).standard_normal(chunks.shape).astype(np.float32)).cuda()
    out = []
    for keep in (True, False):
        U = _pack(mcg, [synth.make_field(dims, 0.7, 2)], dims)
        G = mcg.mcg_pack_gauge(torch.from_numpy(synth.random_gauge(dims, 8)).unsqueeze(0).cuda(), dims)
        torch.cuda.synchronize()
        assert fn(Wd.data_ptr(), Wl.data_ptr() if lo else None, U.data_ptr(), G.data_ptr(), ctypes.byref(g), 1, keep, None) == 0
        torch.cuda.synchronize()
        out.append((U.cpu(), G.cpu()))
    for a, b in zip(*out):
        assert a.isnan().any() and torch.equal(a.isnan(), b.isnan())
        assert float((a - b).nan_to_num().abs().max()) < 1e-14


# a field that stops in the chunk in flight when a restart is queued behind it begins again all the same, and sweeps up
# to the phase's cap: each pass takes S sweeps of two chunks, five passes fit
@pytest.mark.parametrize("copies", [1, 3])
def test_restarts_up_to_the_cap(copies):
    from paper_0807_0264_gb300 import mcg

    dims = (4, 4, 4, 6)
    U = _pack(mcg, [synth.make_field(dims, 0.4, 7, gauge=False)], dims)

    def sweeps32(cap, chunk, restart):
        prm = mcg.Params(tol=1e300, max_sweeps=100000, check_every=chunk, fp32_sweeps=cap, fp32_tol=1e-5, fp32_window=1,
                         fp32_restart=restart)
        if copies == 1:
            return mcg.mcg_precondition_fix(U.clone(), mcg.identity_gauge(dims), dims, prm)[0]["sweeps_fp32"]
        rs = mcg.mcg_precondition_fix(torch.cat([U] * copies), mcg.identity_gauge(dims, copies), dims, prm)
        assert len({r["sweeps_fp32"] for r in rs}) == 1
        return rs[0]["sweeps_fp32"]

    S = sweeps32(1000, 20, 0)
    assert 6 <= S < 100, S
    chunk = (2 * S) // 3
    assert chunk < S < 2 * chunk
    assert sweeps32(5 * S, chunk, chunk) == 5 * S


# round-off of long plain FP64 fixes is a random walk: each sweep stores every link twice and the transforms of its ends
# once, ~6e-17 rms together; the bar is twice sqrt(n) of that
@pytest.mark.parametrize("n,seed", [(1000, 3), (3000, 4)])
def test_long_fixes_stay_on_the_gauge_orbit(n, seed):
    from paper_0807_0264_gb300 import mcg

    dims = (6, 4, 6, 8)
    U0 = synth.make_field(dims, 2.0, seed)
    U, G = _pack(mcg, [U0], dims), mcg.identity_gauge(dims)
    mcg.mcg_fix(U, G, dims, mcg.Params(tol=-1e300, max_sweeps=n, check_every=50))
    d = oracle.apply_gauge(dims, U0, mcg.mcg_unpack_gauge(G, dims)[0].cpu().numpy()) - mcg.mcg_unpack_links(U, dims)[0].cpu().numpy()
    assert np.sqrt((np.abs(d) ** 2).mean()) < 2 * 6e-17 * np.sqrt(n)


# links whose output gradients differ by many orders: a term keeps its own precision, as in FP64 arithmetic, where the
# large ones near it do not reach it (rho = 0) or reach it by a small weight
@pytest.mark.parametrize("eps", [1.0, -0.25])
@pytest.mark.parametrize("rho", [0.0, 1e-18, 1e-9])
def test_smear_backward_of_unequal_gradients(eps, rho):
    from paper_0807_0264_gb300 import mcg

    dims, rng = (4, 2, 6, 4), np.random.default_rng(9)
    U = synth.make_field(dims, 0.7, 9)
    G = rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape)
    G *= 10.0 ** rng.integers(-6, 7, U.shape[:2] + (1, 1))
    got = mcg.mcg_smear_backward_step(_pack(mcg, [U], dims), _pack(mcg, [G], dims), dims, rho, eps)
    got = mcg.mcg_unpack_links(got, dims)[0].cpu().numpy()
    ref = oracle.smear_step_backward(dims, U, G, rho, eps)
    # per link: ~30 roundings of 1.1e-16 of its own gradient, and of the weighted sum of up to 24 staples of its neighbours
    own = np.abs(G).max(axis=(-2, -1))
    bar = 5e-15 * own + 24 * 5e-15 * rho * np.abs(G).max()
    assert (np.abs(got - ref).max(axis=(-2, -1)) < bar).all()


# the two block orders of stout steps: tiles without and with a ragged last one (64 and 1 000 sites of a parity), and
# lattices whose tiles would be too empty (8, 72, 120), several fields per call.  FP64: 2e-14 per step; FP32: ~150
# roundings of 6e-8 per link and step
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 2), (6, 6, 2, 2), (4, 6, 10, 2), (10, 10, 10, 2)])
def test_block_orders_of_stout_steps(dims):
    from paper_0807_0264_gb300 import mcg

    Us = [synth.make_field(dims, 0.7, s) for s in range(3)]
    Ud = _pack(mcg, Us, dims)
    S = mcg.mcg_unpack_links(mcg.mcg_smear(Ud, dims, 0.1, 1.0, 2), dims).cpu().numpy()
    S32 = mcg.mcg_unpack_links(mcg.mcg_smear(mcg.mcg_convert(Ud, mcg.F32), dims, 0.1, 1.0, 2), dims).cpu().numpy()
    for U, s, s32 in zip(Us, S, S32):
        ref = oracle.smear(dims, U, 0.1, 1.0, 2)
        assert np.abs(s - ref).max() < 4e-14 and np.abs(s32 - ref).max() < 2e-5


# the other block order, a kind's sites in whole warps or not (200 and 20 fields: the rule's other side), stout and
# over-improved.  FP64: 2e-14 per step; FP32: ~500 roundings of 6e-8 per link and step
@pytest.mark.parametrize("eps,rho", [(1.0, 0.1), (-0.25, 0.06)])
@pytest.mark.parametrize("dims,copies", [((2, 2, 2, 2), 1), ((2, 2, 2, 2), 67), ((6, 6, 2, 2), 2), ((6, 6, 2, 2), 22), ((6, 6, 6, 2), 7)])
def test_rows_of_whole_warps(dims, copies, eps, rho):
    from paper_0807_0264_gb300 import mcg

    Us = [synth.make_field(dims, 0.7, s) for s in range(3)]
    Ud = _pack(mcg, Us * copies, dims)
    S = mcg.mcg_unpack_links(mcg.mcg_smear(Ud, dims, rho, eps, 2), dims).cpu().numpy()
    S32 = mcg.mcg_unpack_links(mcg.mcg_smear(mcg.mcg_convert(Ud, mcg.F32), dims, rho, eps, 2), dims).cpu().numpy()
    refs = [oracle.smear(dims, U, rho, eps, 2) for U in Us]
    for k in range(3 * copies):
        assert np.abs(S[k] - refs[k % 3]).max() < 4e-14 and np.abs(S32[k] - refs[k % 3]).max() < 6e-5


# batches whose scratch is more than its share of the free memory go a few fields at a time: the same bits
@pytest.mark.parametrize("eps,rho", [(1.0, 0.1), (-0.25, 0.06)])
def test_smearing_of_batches_beyond_the_scratch_share(eps, rho):
    from paper_0807_0264_gb300 import mcg

    dims, nf = (8, 8, 8, 8), 37
    U = torch.cat([_pack(mcg, [synth.make_field(dims, 0.7, s) for s in range(2)], dims)] * 19)[:nf].contiguous()
    G = torch.randn(U.shape, dtype=U.dtype, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5))
    step, back = mcg.mcg_smear(U, dims, rho, eps, 1), mcg.mcg_smear_backward_step(U, G, dims, rho, eps)
    outs = [torch.empty_like(U), torch.empty_like(U)]
    del outs[1]  # room in the caller's allocator for the gradient
    torch.cuda.synchronize()
    mcg.mcg_release()
    free = torch.cuda.mem_get_info()[0] - (240 << 20)
    assert free > 0
    fill = torch.empty(free, dtype=torch.uint8, device="cuda")  # leaves 240 MB: a share of 60 MB, a copy takes 87
    try:
        mcg.mcg_smear(U, dims, rho, eps, 1, outs[0])
        assert torch.equal(outs[0], step)
        assert torch.equal(mcg.mcg_smear_backward_step(U, G, dims, rho, eps), back)
    finally:
        del fill
        mcg.mcg_release()
        torch.cuda.empty_cache()
