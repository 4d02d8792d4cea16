"""Sizes and inputs at which the fixed-point hops, the 256-site block solver
and the blocked LU can go wrong, against the oracle, the FP64 form of the same
operator or torch's dense LU."""
import ctypes
import time

import numpy as np
import pytest
import torch

import paper_1204_1306_gb300 as ps
from oracle import dirac, estimator, gauge, lattice
from oracle.gamma import GAMMA
from tests import seeded
from tests.gpu_util import canonical, get_links, native, rel_err, set_links

pytestmark = pytest.mark.gpu


def _ctx(dims, block, seed=11, kappa=0.15, eps=0.4):
    ctx = ps.psms_create(dims, block, kappa, 1)
    ps.psms_gauge_init(ctx, 0, eps, seed)
    return ctx, gauge.generate_links(dims, eps, seed)


def _apply(ctx, nat, op, graph=False):
    """D psi; graph: under stream capture, where the FP64 form of the hops runs."""
    out = torch.zeros_like(nat)
    if not graph:
        ps.psms_dw_apply(ctx, 0, op, nat, out, ps.PREC_F64)
        torch.cuda.synchronize()
        return out.view(torch.float64)
    ps.psms_autotune(ctx, False)  # no timing runs inside the capture
    s = torch.cuda.Stream()
    ps.psms_set_stream(ctx, s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        ps.psms_dw_apply(ctx, 0, op, nat, out, ps.PREC_F64)
    ps.psms_set_stream(ctx, None)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    return out.view(torch.float64)


# (below and above the split into directions; V/2 not a multiple of a CTA; odd block counts)
@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((6, 4, 4, 2), (2, 2, 2, 2)),
                                        ((12, 12, 12, 12), (4, 4, 4, 4)), ((16, 8, 16, 12), (8, 2, 4, 4))])
@pytest.mark.parametrize("op", [ps.OP_FULL, ps.OP_BLOCKS, 1])
def test_fixed_point_hops_against_the_fp64_form(dims, block, op):
    ctx, _ = _ctx(dims, block)
    nat = native(ctx, seeded.spinor(dims, 3))
    a, b = _apply(ctx, nat, op), _apply(ctx, nat, op, graph=True)
    # each site is a sum of 192 products; both forms round to a few 2^-53 of its largest terms
    assert float((a - b).abs().max() / b.abs().max()) < 64 * 2.0 ** -53


@pytest.mark.parametrize("prec,tol,warm", [(ps.PREC_F64, 64 * 2.0 ** -53, True), (ps.PREC_F64, 64 * 2.0 ** -53, False),
                                           (ps.PREC_F32, 0.0, True), (ps.PREC_BF16, 0.0, True)])
def test_capture_with_the_default_settings(prec, tol, warm):
    """An operator call is captured with autotuning on, after a warm-up call and
    without one (FP64: the captured call runs another form than the warm-up; the
    other precisions allocate their links in the warm-up)."""
    dims = (8, 8, 8, 8)
    ctx, _ = _ctx(dims, (4, 4, 4, 4))
    nat = native(ctx, seeded.spinor(dims, 9), prec)
    typ = {ps.PREC_F64: torch.float64, ps.PREC_F32: torch.float32, ps.PREC_BF16: torch.bfloat16}[prec]
    out = torch.zeros_like(nat)

    def call():
        ps.psms_dw_apply(ctx, 0, ps.OP_FULL, nat, out, prec)

    if warm:
        call()
        torch.cuda.synchronize()
    s = torch.cuda.Stream()
    ps.psms_set_stream(ctx, s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    ps.psms_set_stream(ctx, None)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    got = out.view(typ).double()
    call()
    torch.cuda.synchronize()
    ref = out.view(typ).double()
    assert float(ref.abs().max()) > 0.1
    assert float((got - ref).abs().max()) <= tol * float(ref.abs().max())


def test_hops_without_room_for_the_converted_input():
    """All but 256 MB of the device is held, so that the 407 MB copy of the input
    does not fit: the sites are converted as they are read, to the same bits."""
    dims = (64, 32, 32, 32)
    ctx = ps.psms_create(dims, (4, 4, 4, 4), 0.15, 1)
    ps.psms_gauge_init(ctx, 0, 0.4, 11)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    nat = torch.randn(int(np.prod(dims)) * 24, dtype=torch.float64, device="cuda", generator=g)
    out = torch.zeros_like(nat)
    ps.psms_dw_apply(ctx, 0, 3, nat, out, ps.PREC_F64)  # one block: makes the copy of the links, not of the input
    torch.cuda.synchronize()
    held = ps.psms_scratch_bytes(ctx)
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (256 << 20), dtype=torch.uint8, device="cuda")
    ps.psms_dw_apply(ctx, 0, ps.OP_FULL, nat, out, ps.PREC_F64)
    torch.cuda.synchronize()
    assert ps.psms_scratch_bytes(ctx) == held
    got = out.cpu()
    del fill
    torch.cuda.empty_cache()
    ps.psms_dw_apply(ctx, 0, ps.OP_FULL, nat, out, ps.PREC_F64)
    torch.cuda.synchronize()
    assert ps.psms_scratch_bytes(ctx) > held
    assert torch.equal(out.cpu(), got)


def test_hops_alternating_between_streams():
    dims = (16, 16, 16, 16)  # the form that keeps the input in scratch
    ctx, _ = _ctx(dims, (4, 4, 4, 4))
    nats = [native(ctx, seeded.spinor(dims, k)) for k in range(4)]
    refs = [_apply(ctx, nat, ps.OP_FULL) for nat in nats]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [[torch.zeros_like(nat) for nat in nats] for _ in range(8)]
    torch.cuda.synchronize()
    for row in outs:
        for k, nat in enumerate(nats):
            ps.psms_set_stream(ctx, streams[k % 2])
            ps.psms_dw_apply(ctx, 0, ps.OP_FULL, nat, row[k], ps.PREC_F64)
    ps.psms_set_stream(ctx, None)
    torch.cuda.synchronize()
    for row in outs:
        for out, ref in zip(row, refs):
            assert torch.equal(out.view(torch.float64), ref)


def test_hops_on_streams_that_are_destroyed_at_once():
    """A stream destroyed with a hop in flight, and the next one, which may get
    the same handle: the second call waits for the first one's scratch."""
    dims = (16, 16, 16, 16)
    ctx, _ = _ctx(dims, (4, 4, 4, 4))
    nats = [native(ctx, seeded.spinor(dims, k)) for k in range(2)]
    refs = [_apply(ctx, nat, ps.OP_FULL) for nat in nats]
    outs = [torch.zeros_like(nats[k % 2]) for k in range(16)]
    torch.cuda.synchronize()
    rt = torch.cuda.cudart()
    for k, out in enumerate(outs):
        h = ctypes.c_void_p()
        assert int(rt.cudaStreamCreate(ctypes.addressof(h))) == 0
        ps.psms_set_stream(ctx, h.value)
        ps.psms_dw_apply(ctx, 0, ps.OP_FULL, nats[k % 2], out, ps.PREC_F64)
        assert int(rt.cudaStreamDestroy(h.value)) == 0
    ps.psms_set_stream(ctx, None)
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        assert torch.equal(out.view(torch.float64), refs[k % 2])


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((16, 16, 16, 8), (4, 4, 4, 4))])
@pytest.mark.parametrize("scale", [2.0 ** -1000, 2.0 ** -850, 2.0 ** 850, 2.0 ** 1000])
def test_hops_at_the_ends_of_the_fp64_range(dims, block, scale):
    ctx, _ = _ctx(dims, block)
    nat = native(ctx, seeded.spinor(dims, 4))
    ref = _apply(ctx, nat, ps.OP_FULL)
    big = nat.clone()
    big.view(torch.float64).mul_(scale)  # a power of two: exact
    got = _apply(ctx, big, ps.OP_FULL)
    assert float((got / scale - ref).abs().max() / ref.abs().max()) < 64 * 2.0 ** -53


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((16, 16, 16, 8), (4, 4, 4, 4))])
def test_hops_of_colours_of_different_size(dims, block):
    """The unit field does not mix colours: each keeps the accuracy of FP64."""
    ctx = ps.psms_create(dims, block, 0.15, 1)
    psi = seeded.spinor(dims, 12) * np.array([1.0, 1e-6, 1e-12])
    nat = native(ctx, psi)
    a = canonical(ctx, _apply(ctx, nat, ps.OP_FULL).view(torch.uint8))
    b = canonical(ctx, _apply(ctx, nat, ps.OP_FULL, graph=True).view(torch.uint8))
    for c in range(3):
        assert np.abs(a[..., c] - b[..., c]).max() < 64 * 2.0 ** -53 * np.abs(b[..., c]).max()


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((16, 16, 16, 8), (4, 4, 4, 4))])
def test_hops_of_a_point_source(dims, block):
    """Entries of links next to the unit matrix: each output number is one product."""
    ctx = ps.psms_create(dims, block, 0.15, 1)
    ps.psms_gauge_init(ctx, 0, 1e-6, 13)
    psi = np.zeros(dims + (4, 3), dtype=np.complex128)
    psi[1, 2, 0, 3, 1, 2] = 1.0
    nat = native(ctx, psi)
    a, b = _apply(ctx, nat, ps.OP_FULL), _apply(ctx, nat, ps.OP_FULL, graph=True)
    assert int((b != 0).sum()) > 60
    assert bool(((a - b).abs() <= 4 * 2.0 ** -53 * b.abs()).all())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((16, 16, 16, 8), (4, 4, 4, 4))])
def test_non_finite_spinors_spread_as_in_fp64(dims, block, bad):
    ctx, _ = _ctx(dims, block)
    nat = native(ctx, seeded.spinor(dims, 5))
    nat.view(torch.float64)[2 * 77 + 1] = bad
    a, b = _apply(ctx, nat, ps.OP_FULL), _apply(ctx, nat, ps.OP_FULL, graph=True)
    fin = torch.isfinite(b)
    assert 24 < int((~fin).sum()) <= 9 * 24
    assert torch.equal(fin, torch.isfinite(a))
    assert float((a[fin] - b[fin]).abs().max()) < 64 * 2.0 ** -53 * float(b[fin].abs().max())


def test_copies_of_a_field_follow_its_changes():
    dims, block = (8, 8, 8, 8), (4, 4, 4, 4)
    ctx, _ = _ctx(dims, block)
    nat = native(ctx, seeded.spinor(dims, 6))
    first = _apply(ctx, nat, ps.OP_FULL).clone()
    ps.psms_gauge_sweep(ctx, 0, ps.ACTIVE_ALL, 1, 0, 5.3, 3, 0)
    a, b = _apply(ctx, nat, ps.OP_FULL), _apply(ctx, nat, ps.OP_FULL, graph=True)
    assert float((a - b).abs().max() / b.abs().max()) < 64 * 2.0 ** -53
    assert float((a - first).abs().max()) > 1e-3


# every way to cut 256 sites that the link layout of the block solver treats apart, odd block counts among them
@pytest.mark.parametrize("dims,block", [((4, 4, 4, 4), (4, 4, 4, 4)), ((8, 4, 4, 2), (8, 4, 4, 2)),
                                        ((4, 4, 12, 8), (4, 4, 2, 8)), ((16, 4, 4, 4), (16, 4, 2, 2)),
                                        ((2, 2, 4, 32), (2, 2, 2, 32)), ((32, 4, 2, 4), (32, 2, 2, 2)),
                                        ((12, 4, 4, 4), (4, 4, 4, 4))])
@pytest.mark.parametrize("krylov", [None, ps.SOLVER_CGNR, ps.SOLVER_BICGSTAB])
def test_block_solver_shapes(dims, block, krylov):
    assert int(np.prod(block)) == 256
    ctx, U = _ctx(dims, block, kappa=0.156, eps=0.5)
    if krylov is not None:
        ps.psms_block_krylov(ctx, krylov)
    geom = lattice.Geometry(dims, block)
    b = seeded.spinor(dims, 7)
    nat = native(ctx, b)
    x = torch.zeros_like(nat)
    info = ps.psms_solve(ctx, 0, ps.OP_BLOCKS, nat, x, 1e-13, 20000, ps.PREC_F32)
    assert info["true_residual"] <= 1e-13
    got = canonical(ctx, x)
    r = b - dirac.apply_D(U, got, 0.156, geom, mode="block")
    assert np.sqrt(np.sum(np.abs(r) ** 2) / np.sum(np.abs(b) ** 2)) < 2e-13
    last = geom.n_blocks - 1
    ref = estimator.solve_blocks(U, b, geom, 0.156, [last], 1e-14)
    assert rel_err(dirac.extract_block(got, geom, last), dirac.extract_block(ref, geom, last)) < 1e-11


def test_block_solver_right_hand_sides():
    """A zero block, a block with an even half only, and the iteration cap."""
    dims, block = (8, 4, 4, 4), (4, 4, 4, 4)
    ctx, U = _ctx(dims, block, kappa=0.156, eps=0.5)
    geom = lattice.Geometry(dims, block)
    b = seeded.spinor(dims, 8)
    b[:4] = 0
    b[4:][geom.parity[4:] == 1] = 0
    nat = native(ctx, b)
    x = torch.zeros_like(nat)
    info = ps.psms_solve(ctx, 0, ps.OP_BLOCKS, nat, x, 1e-13, 20000, ps.PREC_F32)
    got = canonical(ctx, x)
    assert info["true_residual"] <= 1e-13 and np.abs(got[:4]).max() == 0.0
    r = b - dirac.apply_D(U, got, 0.156, geom, mode="block")
    assert np.sqrt(np.sum(np.abs(r) ** 2) / np.sum(np.abs(b) ** 2)) < 2e-13
    with pytest.raises(ps.PsmsError) as e:
        ps.psms_solve(ctx, 0, ps.OP_BLOCKS, nat, x, 1e-13, 3, ps.PREC_F32)
    assert e.value.status == 4  # PSMS_ENOCONV


def test_sweep_lists_are_made_once():
    """Both active sets in turn give what a fresh context gives, and a later call
    does not walk over the block on the host again (one block of 2^20 sites)."""
    dims, block = (8, 8, 4, 4), (4, 4, 4, 4)
    ctx, _ = _ctx(dims, block)
    for k, active in enumerate((ps.ACTIVE_ALL, ps.ACTIVE_BLOCKS, ps.ACTIVE_ALL, ps.ACTIVE_BLOCKS)):
        fresh, _ = _ctx(dims, block)
        set_links(fresh, 0, get_links(ctx, 0))
        for c in (ctx, fresh):
            ps.psms_gauge_sweep(c, 0, active, 1, 1, 5.3, 3, 10 * k)
        assert np.array_equal(get_links(ctx, 0), get_links(fresh, 0))

    def calls(n):
        ctx = ps.psms_create((32, 32, 32, 32), (32, 32, 32, 32), 0.15, 1)
        t = []
        for _ in range(n):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ps.psms_gauge_sweep(ctx, 0, ps.ACTIVE_BLOCKS, 0, 0, 5.3, 3, 0)  # no updates: the lists and the projection
            t.append(time.perf_counter() - t0)
        return t

    calls(1)
    first, *later = calls(6)
    assert min(later) < 0.5 * first


@pytest.mark.parametrize("op", [ps.OP_FULL, ps.OP_BLOCKS])
def test_solves_whose_sums_overflow_end(op):
    """Links of 1e25: the FP32 inner iterations' sums become infinite, and the
    solve ends without convergence."""
    dims = (8, 4, 4, 4)
    ctx, U = _ctx(dims, (4, 4, 4, 4))
    set_links(ctx, 0, U * 1e25)
    nat = native(ctx, seeded.spinor(dims, 14))
    with pytest.raises(ps.PsmsError) as e:
        ps.psms_solve(ctx, 0, op, nat, torch.zeros_like(nat), 1e-12, 500, ps.PREC_F32)
    assert e.value.status == 4  # PSMS_ENOCONV


# BiCGStab: the better method; slow; stagnating; without convergence
@pytest.mark.parametrize("kappa,eps", [(0.25, 3.0), (0.2, 0.3), (0.25, 0.3), (0.4, 0.3), (1.0, 0.3), (20.0, 0.3)])
def test_block_bicgstab_gives_way_to_cgnr(kappa, eps):
    """Whatever CGNR solves is solved, with BiCGStab's attempts as the only extra
    cost: 48 iterations at most for each of up to 12 corrections before one fails,
    which they do at once where they are many."""
    dims, block = (8, 4, 4, 4), (4, 4, 4, 4)
    b = seeded.spinor(dims, 7)
    geom = lattice.Geometry(dims, block)
    its = {}
    for krylov in (None, ps.SOLVER_CGNR):
        ctx, U = _ctx(dims, block, seed=3, kappa=kappa, eps=eps)
        if krylov is not None:
            ps.psms_block_krylov(ctx, krylov)
        nat = native(ctx, b)
        x = torch.zeros_like(nat)
        info = ps.psms_solve(ctx, 0, ps.OP_BLOCKS, nat, x, 1e-12, 20000, ps.PREC_F32)
        r = b - dirac.apply_D(U, canonical(ctx, x), kappa, geom, mode="block")
        assert np.sqrt(np.sum(np.abs(r) ** 2) / np.sum(np.abs(b) ** 2)) < 2e-12
        its[krylov] = info["inner_iters"]
    assert its[None] <= its[ps.SOLVER_CGNR] + 2 * 2 * 48  # two blocks, a failure in the first or second correction


@pytest.mark.parametrize("kappa,eps", [(0.4, 0.3), (0.156, 0.5)])
def test_block_iteration_cap_is_that_of_cgnr(kappa, eps):
    """A cap that CGNR meets exactly suffices, one below it does not (one block)."""
    dims = (4, 4, 4, 4)
    ctx, _ = _ctx(dims, dims, seed=3, kappa=kappa, eps=eps)
    nat = native(ctx, seeded.spinor(dims, 7))
    x = torch.zeros_like(nat)
    ps.psms_block_krylov(ctx, ps.SOLVER_CGNR)
    need = ps.psms_solve(ctx, 0, ps.OP_BLOCKS, nat, x, 1e-12, 20000, ps.PREC_F32)["inner_iters"]
    with pytest.raises(ps.PsmsError):
        ps.psms_solve(ctx, 0, ps.OP_BLOCKS, nat, x, 1e-12, need // 3, ps.PREC_F32)
    fresh, _ = _ctx(dims, dims, seed=3, kappa=kappa, eps=eps)
    assert ps.psms_solve(fresh, 0, ps.OP_BLOCKS, nat, x, 1e-12, need, ps.PREC_F32)["true_residual"] <= 1e-12


def test_block_level_is_as_accurate_as_with_cgnr():
    """The estimates' error against a tighter solve, at the tolerance that two
    BiCGStab corrections of 1e-6 may just meet."""
    ctx = ps.psms_create((8, 8, 8, 8), (4, 4, 4, 4), 0.156, 2)
    ps.psms_gauge_init(ctx, 0, 0.5, 21)
    ps.psms_gauge_copy(ctx, 1, 0)
    ps.psms_gauge_sweep(ctx, 1, ps.ACTIVE_BLOCKS, 1, 1, 5.3, 22, 0)

    def level(tol):
        return np.asarray(ps.psms_logdet_ratio(ctx, ps.LEVEL_BLOCK, 0, 1, 12, ps.EST_INTERP, 23, 7, tol, ps.PREC_F32))

    got = level(1e-13)
    ps.psms_block_krylov(ctx, ps.SOLVER_CGNR)
    ref = level(1e-14)
    # |x|^2 of 3072 numbers of unit variance: 4 x 3072 roundings of 2^-53 at most, 1.4e-12; a residual of 1e-13 / 16
    # moves it by 2 |D_b^-1 r| |x| / sqrt(3072) = 2 |D_b^-1| |b| 6e-15 < 2 x 2 x 110 x 6e-15 = 2.7e-12
    assert np.sqrt(np.mean((got - ref) ** 2)) < 4e-12


# 16 sites (one sub-panel row per thread), 64, 256, and 512 sites (the tall panels)
@pytest.mark.parametrize("dims,block", [((4, 4, 4, 2), (2, 2, 2, 2)), ((4, 4, 4, 4), (4, 4, 2, 2)),
                                        ((4, 4, 4, 8), (4, 4, 4, 4)), ((8, 4, 4, 4), (8, 4, 4, 4))])
def test_lu_sizes_against_torch(dims, block):
    kappa = 0.15
    ctx, U = _ctx(dims, block, kappa=kappa)
    geom = lattice.Geometry(dims, block)
    got = ps.psms_block_logdet(ctx, 0)
    for b in sorted({0, geom.n_blocks - 1}):
        ref = _dense_logdet(dirac.extract_block(U, geom, b), block, kappa)
        assert abs(got[b] - ref) < 1e-11 * abs(ref)


def _dense_logdet(Ub, block, kappa):
    """ln |det D_b| from torch's LU of A - D_oe D_eo / A, the hops written into a dense matrix."""
    A = 1.0 / (2.0 * kappa)
    n = int(np.prod(block))
    u = torch.from_numpy(np.ascontiguousarray(Ub)).cuda()
    D = torch.zeros(n, 4, 3, n, 4, 3, dtype=torch.complex128, device="cuda")
    g = torch.arange(n, device="cuda").reshape(block)
    for mu in range(4):
        x, y = g.narrow(mu, 0, block[mu] - 1).reshape(-1), g.narrow(mu, 1, block[mu] - 1).reshape(-1)
        w = u[..., mu, :, :].reshape(n, 3, 3)[x]
        gm = torch.from_numpy(np.asarray(GAMMA[mu], dtype=np.complex128)).cuda()
        one = torch.eye(4, dtype=torch.complex128, device="cuda")
        for t, src, dst, m in ((-1.0, y, x, w), (1.0, x, y, w.conj().transpose(-1, -2))):
            D[dst, :, :, src, :, :] += -0.5 * (one + t * gm)[None, :, None, :, None] * m[:, None, :, None, :]
    par = torch.from_numpy((np.indices(block).sum(0) % 2).reshape(-1)).cuda()
    o, e = torch.nonzero(par == 1).reshape(-1), torch.nonzero(par == 0).reshape(-1)
    D = D.reshape(n, 12, n, 12)
    oe, eo = D[o][:, :, e].reshape(6 * n, 6 * n), D[e][:, :, o].reshape(6 * n, 6 * n)
    M = A * torch.eye(6 * n, dtype=torch.complex128, device="cuda") - (oe @ eo) / A
    return 6 * n * np.log(A) + torch.linalg.slogdet(M).logabsdet.item()
