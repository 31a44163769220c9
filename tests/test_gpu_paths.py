"""GPU tests of the kernels' alternative paths at the sizes where they can go
wrong: remainders, wrap-around on the smallest extents, both sides of a rule."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_helpers import hop_ref, rel, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    return require_cuda()


def on_device(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def exchanges_rows(block):
    m = block.copy()
    for k in range(6):
        if np.abs(m[k + 1:, k]).max(initial=0.0) > np.abs(m[k, k]):
            return True
        m[k + 1:] -= np.outer(m[k + 1:, k] / m[k, k], m[k])
    return False


@pytest.mark.parametrize("dims,kind,kappa,csw", [
    ((2, 2, 2, 2), "haar", 0.13, 1.0),
    ((4, 2, 6, 2), "haar", 0.3, 3.0),      # strong field: rows have to be exchanged in the inversion
    ((4, 6, 4, 10), "smooth", 0.135, 1.0),  # 480 sites per parity: blocks of 64 and of 32 sites
    ((6, 10, 2, 14), "haar", 0.25, 2.0),
])
def test_clover_build_and_inverse(lq, dims, kind, kappa, csw):
    """A and A^{-1} against the oracle's A and its LAPACK inverse in FP64 (a
    backward-stable inversion of a 6x6 block is off by a few eps cond), and
    each rounded copy against the FP64 result (one rounding of the operator,
    input and output)."""
    U = synth.gauge_field(dims, kind, 3, eps=0.5)
    A = oracle.clover(U, kappa, csw)
    blocks = np.stack([A[..., :6, :6], A[..., 6:, 6:]]).reshape(-1, 6, 6)
    if kind == "haar" and kappa > 0.2:  # partial pivoting exchanges rows in some blocks, not in all
        assert 0 < np.mean([exchanges_rows(b) for b in blocks]) < 1
    cond = np.linalg.cond(blocks).max()
    psi = synth.gaussian_spinor(dims, 4)
    want = {0: np.einsum("...ab,...b->...a", A, psi.reshape(psi.shape[:4] + (12,))),
            1: np.linalg.solve(A, psi.reshape(psi.shape[:4] + (12, 1)))[..., 0]}
    lat = lq.Lattice(dims)
    lat.gauge_load(on_device(U))
    lat.clover_compute(kappa, csw)
    par = np.indices(psi.shape[:4]).sum(axis=0) % 2
    for prec, eps in (("f64", 2.2e-16), ("f32", 1.2e-7), ("f16", 2.0 ** -10), ("bf16", 2.0 ** -7)):
        for inverse in (0, 1):
            out = lat.canonical_spinor()
            for p in (0, 1):
                fin, fout = lat.new_field(prec), lat.new_field(prec)
                lat.pack(fin, on_device(psi), p, prec)
                lat.clover_apply(fout, fin, p, inverse, prec)
                lat.unpack(out, fout, p, prec)
            lat.sync()
            got = out.cpu().numpy().reshape(want[0].shape)
            for p in (0, 1):
                g, w = got[par == p], want[inverse][par == p]
                size = np.linalg.norm(A[par == p] if not inverse else np.linalg.inv(A[par == p]), axis=(-2, -1))
                tol = 8 * eps + (50 * 2.2e-16 * cond if inverse else 0.0)
                # per site: against the size of the operator times the input
                err = np.linalg.norm(g - w, axis=-1) / (size * np.linalg.norm(psi.reshape(par.shape + (12,))[par == p], axis=-1))
                assert err.max() < tol, (prec, inverse, p, err.max(), tol)


@pytest.mark.parametrize("dims,nrhs,recon", [
    ((2, 2, 2, 2), 1, 12),      # 8 sites per parity: most lanes idle, every neighbour wraps
    ((4, 2, 6, 6), 3, 18),      # 144 sites: a last block of 16
    ((8, 8, 8, 8), 1, 12),
    ((6, 10, 14, 4), 5, 12),    # 8400 site-rhs: past the FP64 line, below the reducing one
    ((8, 16, 16, 16), 1, 12),   # 16384: the last size of the plain launches
    ((8, 16, 16, 18), 1, 12),   # the first past it
])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "bf16links", "f16spinors", "bf16"])
def test_small_launch_kernel_is_bit_identical(lq, dims, nrhs, recon, prec):
    """The warp-per-direction kernel of small launches against the gathering
    kernel (selected by a block of 96 threads): every operator, both
    directions, with and without a clover term, bit for bit; the hopping term
    against the oracle as well."""
    import torch
    U = synth.gauge_field(dims, "smooth", 5, eps=0.5)
    psi = np.stack([synth.gaussian_spinor(dims, 6 + r) for r in range(nrhs)])
    lat = lq.Lattice(dims, precisions=("f64", "f32", prec), recon=recon, max_nrhs=nrhs)
    lat.gauge_load(on_device(U))
    for csw in (0.0, 1.0):
        lat.clover_compute(0.13, csw)
        for op in (lq.OP_HOP, lq.OP_SCHUR, lq.OP_FULL):
            full = op == lq.OP_FULL
            fin = lat.new_field(prec, nrhs, full)
            lat.pack(fin, on_device(psi), -1 if full else 1, prec, nrhs)
            for dag in (False, True):
                out = []
                for block in (128, 96):
                    lq.lqcd_tune_set(lat.ctx, prec, (block,) * 4)
                    f = torch.zeros_like(fin)
                    lat.dslash(f, fin, 1 if op == lq.OP_SCHUR else 0, 0.13, csw, op, dag, prec, nrhs)
                    lat.sync()
                    out.append(f)
                assert torch.equal(*out), (csw, op, dag)
    if prec == "f64" and nrhs > 1:
        fin, fout = lat.new_field(prec, nrhs), lat.new_field(prec, nrhs)
        lat.pack(fin, on_device(psi), 1, prec, nrhs)
        lq.lqcd_tune_set(lat.ctx, prec, (128,) * 4)
        lat.dslash(fout, fin, 0, prec=prec, nrhs=nrhs)
        got = lat.canonical_spinor(nrhs)
        lat.unpack(got, fout, 0, prec, nrhs)
        lat.sync()
        for r in range(nrhs):
            assert rel(got[r].cpu().numpy(), hop_ref(U, psi[r], dims, 0)) < 1e-13


@pytest.mark.parametrize("dims,inner", [((2, 2, 2, 2), "f64"), ((4, 2, 6, 6), "f32"), ((8, 8, 8, 8), "f16spinors"),
                                        ((8, 16, 16, 12), "f32")])
@pytest.mark.parametrize("graph", [0, 1])
def test_small_solves(lq, dims, inner, graph):
    """Solves whose every launch is small (reducing epilogues, captured and
    not): the oracle's true residual, and the iterates of the gathering
    kernel's solve (fields bit-identical, global sums regrouped)."""
    import torch
    U = synth.gauge_field(dims, "smooth", 7, eps=0.5)
    b = synth.gaussian_spinor(dims, 8)
    lat = lq.Lattice(dims, precisions=("f64", "f32"), stream=torch.cuda.Stream())
    lat.gauge_load(on_device(U))
    lat.clover_compute(0.12, 1.0)
    A = oracle.clover(U, 0.12, 1.0)
    xs = []
    for block in (128, 96):
        for prec in {"f64", "f32", inner}:
            lq.lqcd_tune_set(lat.ctx, prec, (block,) * 4)
        x, bd = lat.canonical_spinor(), on_device(b)
        torch.cuda.synchronize()
        _, st = lat.solve(x, bd, 1e-10, inner_prec=inner, use_graph=graph)
        xs.append(x.cpu().numpy())
        assert oracle.true_residual(U, A, 0.12, b, xs[-1]) <= 1e-10
    assert rel(xs[0], xs[1]) < 1e-8  # both within 1e-10 residual of the solution, |M^-1| |M| well below 100


@pytest.mark.parametrize("dims,block,recon,csw", [
    ((8, 8, 8, 8), (4, 4, 4, 4), 18, 1.0),    # the constant-extent kernel
    ((8, 8, 8, 8), (4, 4, 4, 2), 12, 1.0),    # extents from the arguments
    ((4, 12, 8, 4), (2, 6, 4, 2), 12, 1.0),   # 96 sites a block: a whole number of warps, fewer than the CTA's most
    ((12, 12, 4, 4), (6, 6, 2, 2), 18, 1.0),  # 144: idle lanes
    ((8, 8, 8, 8), (4, 4, 4, 4), 12, 0.0),    # no clover term
    ((8, 16, 16, 40), (4, 4, 4, 4), 12, 1.0),  # more blocks of a colour than SMs: two on one
    ((8, 8, 12, 16), (2, 2, 2, 2), 18, 1.0),   # the same, 16 sites a block
])
def test_sap_block_kernel(lq, dims, block, recon, csw):
    """SAP of blocks of at most 256 sites against the oracle (FP32 sums of
    about 2000 products a site, 6e-8 each, through nmr ncycle steps: 1e-5
    bounds it generously), after other fields went through the same context."""
    U = [synth.gauge_field(dims, "smooth", 11 + k, eps=0.5) for k in range(2)]
    r = synth.gaussian_spinor(dims, 12)
    lat = lq.Lattice(dims, precisions=("f64", "f32"), recon=recon)
    for u in U:  # the second field's clover term must be the one that is used
        lat.gauge_load(on_device(u))
        lat.clover_compute(0.13, csw)
        fr, fz = lat.new_field("f32", full=True), lat.new_field("f32", full=True)
        lat.pack(fr, on_device(r), -1, "f32")
        lat.sap_apply(fz, fr, block, 2, 3)
        z = lat.canonical_spinor()
        lat.unpack(z, fz, -1, "f32")
        lat.sync()
    A = oracle.clover(U[1], 0.13, csw) if csw else None
    assert rel(z.cpu().numpy(), oracle.sap(U[1], A, 0.13, r, block, 2, 3)) < 1e-5


def test_sap_solves_in_turn(lq):
    """Flexible solves with SAP one after the other on one context, the block
    shape, the field and the solver changing between them: each takes the
    iterations of a fresh context."""
    import torch
    dims = (8, 8, 8, 8)
    b = synth.gaussian_spinor(dims, 13)
    old = lq.Lattice(dims, precisions=("f64", "f32"), gcr_nkrylov=20)
    for seed, block, solver in ((14, (4, 4, 4, 4), lq.SOLVER_FGCR), (15, (4, 4, 4, 4), lq.SOLVER_FGMRES_DR),
                                (15, (4, 4, 2, 4), lq.SOLVER_FGCR), (14, (4, 4, 4, 4), lq.SOLVER_FGCR)):
        U = synth.gauge_field(dims, "smooth", seed, eps=0.5)
        A = oracle.clover(U, 0.13, 1.0)
        its = []
        for lat in (old, lq.Lattice(dims, precisions=("f64", "f32"), gcr_nkrylov=20)):
            lat.gauge_load(on_device(U))
            lat.clover_compute(0.13, 1.0)
            lat.set_sap(block, 2, 4)
            x = lat.canonical_spinor()
            _, st = lat.solve(x, on_device(b), 1e-10, solver=solver, inner_prec="f32", nkrylov=20)
            its.append(st["iterations"])
            assert oracle.true_residual(U, A, 0.13, b, x.cpu().numpy()) <= 1e-10
        assert its[0] == its[1]


@pytest.mark.parametrize("scale", [1.0, 1e-18, 1e17, "mixed"])
@pytest.mark.parametrize("batch", [1, 3])
def test_training_loss(lq, scale, batch):
    """The loss against FP64 sums over the network's own output, for
    components whose squares FP32 holds and for ones that it does not (2^-46
    for each sum; the division and the mean stay in FP64)."""
    import torch
    dims, channels = (4, 2, 6, 6), (1, 3, 1)
    lat = lq.Lattice(dims, precisions=("f64", "f32"))
    lat.gauge_load(on_device(synth.gauge_field(dims, "smooth", 21, eps=0.5)))
    net = lq.Net(lat, channels, bf16=True, max_batch=batch)
    rng = np.random.default_rng(22)
    net.set_weights((0.1 * (rng.standard_normal(net.num_weights) + 1j * rng.standard_normal(net.num_weights))).astype(np.complex64))
    shape = (batch, dims[3], dims[2], dims[1], dims[0], 4, 3)
    r, e = ((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) for _ in range(2))
    if scale == "mixed":  # zeros, and sixteen orders of magnitude on both sides of one
        s = 10.0 ** rng.integers(-16, 17, size=shape)
        s[rng.random(shape) < 0.2] = 0.0
        r, e = r * s, e * s
    else:
        r, e = r * scale, e * scale
    r, e = on_device(r.astype(np.complex64)), on_device(e.astype(np.complex64))
    y = torch.empty_like(r)
    net.forward(y, r, batch)
    lat.sync()
    flat = lambda t: torch.view_as_real(t).reshape(batch, -1).cpu().numpy()
    d = (flat(y) - flat(e)).astype(np.float64)  # the difference is taken in FP32
    want = np.mean((d ** 2).sum(1) / (flat(e).astype(np.float64) ** 2).sum(1))
    assert abs(net.train_step(r, e, batch, lr=0.0) / want - 1.0) < 1e-12


@pytest.mark.parametrize("c", ["0x1.64fa88p+0", "0x1.fbaef8p+0"])
def test_training_loss_of_a_constant_target(lq, c):
    """Every component of the target is the same number, so that every thread's
    96 additions round alike and their errors do not average out.  A loss of
    FP64 sums of positive terms: at most 30 roundings of 2^-53 each in a sum
    (a thread's sum, the block's tree, the blocks) and the division."""
    import math
    import torch
    dims = (16, 16, 16, 16)
    lat = lq.Lattice(dims, precisions=("f64", "f32"))
    lat.gauge_load(on_device(synth.gauge_field(dims, "smooth", 23, eps=0.5)))
    net = lq.Net(lat, (1, 3, 1), bf16=True, max_batch=1)
    rng = np.random.default_rng(24)
    net.set_weights((0.1 * (rng.standard_normal(net.num_weights) + 1j * rng.standard_normal(net.num_weights))).astype(np.complex64))
    shape = (1, dims[3], dims[2], dims[1], dims[0], 4, 3)
    c = float.fromhex(c)
    r = on_device((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64))
    e = torch.full(shape, complex(c, c), dtype=torch.complex64, device="cuda")
    y = torch.empty_like(r)
    net.forward(y, r, 1)
    lat.sync()
    d = (torch.view_as_real(y) - torch.view_as_real(e)).reshape(-1).cpu().numpy().astype(np.float64)
    want = math.fsum(d * d) / (d.size * c * c)  # squares of 24-bit numbers and the products are exact
    assert abs(net.train_step(r, e, 1, lr=0.0) / want - 1.0) < 2 * 31 * 2.0 ** -53


@pytest.mark.parametrize("prec", ["f16spinors", "f16"])
@pytest.mark.parametrize("block", [128, 96])
def test_hop_reads_subnormal_halves(lq, prec, block):
    """A site whose components span more than FP16's normal range: with unit
    links colour 1 carries only values that are subnormal in units of the
    site's norm, and one step of that grid is 2^-24 (flushed to zero they
    would be 2^-15 off)."""
    dims = (4, 4, 4, 4)
    U = np.zeros((4, 4, 4, 4, 4, 3, 3), dtype=complex)
    U[...] = np.eye(3)
    psi = np.zeros((4, 4, 4, 4, 4, 3), dtype=complex)
    psi[1, 2, 1, 3, :, 0] = 1.0 + 0.5j  # t + z + y + x odd
    psi[1, 2, 1, 3, :, 1] = np.array([1, -2, 5, 11]) * 2.0 ** -18 + 1j * np.array([3, 7, -1, 2]) * 2.0 ** -20
    lat = lq.Lattice(dims, precisions=("f64", "f32", prec))
    lat.gauge_load(on_device(U))
    lq.lqcd_tune_set(lat.ctx, prec, (block,) * 4)
    fin, fout = lat.new_field(prec), lat.new_field(prec)
    lat.pack(fin, on_device(psi), 1, prec)
    lat.dslash(fout, fin, 0, prec=prec)
    out = lat.canonical_spinor()
    lat.unpack(out, fout, 0, prec)
    lat.sync()
    got, want = out.cpu().numpy()[..., 1], hop_ref(U, psi, dims, 0)[..., 1]
    norm = np.abs(hop_ref(U, psi, dims, 0)).max()
    assert np.abs(want).max() > 2.0 ** -17 * norm  # well above a step, far below the normal range
    assert np.abs(got - want).max() < 2.0 ** -23 * norm


@pytest.mark.parametrize("inner", ["f32", "f16spinors", "f16"])
@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("check,every,maxiter", [(10, 0, 25), (30, 0, 60), (30, 7, 33), (1, 2, 5)])
def test_deferred_solution_updates(lq, inner, graph, check, every, maxiter):
    """Two right-hand sides of 65536 sites take the deferred x (ring of ten or
    twenty directions: wrapped, cut short by a replacement or by maxiter), one
    the fused update; the steps are the same, so the iterates are equal."""
    import torch
    dims = (16, 16, 16, 32)
    lat = lq.Lattice(dims, precisions=("f64", "f32", inner), max_nrhs=2, stream=torch.cuda.Stream())
    lat.gauge_load(on_device(synth.gauge_field(dims, "smooth", 31, eps=0.5)))
    lat.clover_compute(0.13, 1.0)
    b = on_device(np.stack([synth.gaussian_spinor(dims, 32 + r) for r in range(2)]))
    x2, x1 = torch.zeros_like(b), torch.zeros_like(b)
    torch.cuda.synchronize()
    kw = dict(raise_on_error=False, inner_prec=inner, use_graph=graph, check_interval=check, reliable_interval=every,
              reliable_delta=0.0, maxiter=maxiter)
    lat.solve(x2, b, 1e-30, nrhs=2, **kw)
    for r in range(2):
        lat.solve(x1[r], b[r], 1e-30, nrhs=1, **kw)
    assert torch.equal(x1, x2)


def test_deferred_solve(lq):
    """A deferred solve whose right-hand sides converge at different times."""
    import torch
    dims = (16, 16, 16, 32)
    U = synth.gauge_field(dims, "smooth", 33, eps=0.5)
    lat = lq.Lattice(dims, precisions=("f64", "f32"), max_nrhs=3)
    lat.gauge_load(on_device(U))
    lat.clover_compute(0.125, 1.0)
    A = oracle.clover(U, 0.125, 1.0)
    b = np.stack([synth.gaussian_spinor(dims, 34), np.zeros((32, 16, 16, 16, 4, 3), complex), synth.gaussian_spinor(dims, 35)])
    b[2, 1:] = 0.0
    x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
    lat.solve(x, on_device(b), 1e-10, nrhs=3, inner_prec="f16spinors")
    assert not x[1].any()
    for r in (0, 2):
        assert oracle.true_residual(U, A, 0.125, b[r], x[r].cpu().numpy()) <= 1e-10


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((4, 2, 6, 6), 3), ((8, 4, 8, 10), 2)])  # 8, 144, 1280 sites a parity
@pytest.mark.parametrize("prec,eps", [("f64", 0.0), ("f32", 2.0 ** -24), ("f16", 2.0 ** -10), ("bf16spinors", 2.0 ** -7)])
def test_pack_and_unpack(lq, dims, nrhs, prec, eps):
    """Canonical spinors to internal fields and back, one parity and both, from
    host and device: each component within the storage's rounding of the site's
    largest, untouched sites of a one-parity unpack left alone."""
    import torch
    psi = np.stack([synth.gaussian_spinor(dims, 41 + r) for r in range(nrhs)])
    big = np.abs(psi).max(axis=(-2, -1), keepdims=True)
    par = np.indices(psi.shape[1:5]).sum(axis=0) % 2
    lat = lq.Lattice(dims, precisions=("f64", "f32", prec), max_nrhs=nrhs)
    for parity in (-1, 0, 1):
        for host in (False, True):
            f = lat.new_field(prec, nrhs, parity < 0)
            src = torch.from_numpy(psi) if host else on_device(psi)
            lat.pack(f, src, parity, prec, nrhs)
            out = torch.full(psi.shape, 7.0, dtype=torch.complex128, device="cpu" if host else "cuda")
            lat.unpack(out, f, parity, prec, nrhs)
            lat.sync()
            got = out.cpu().numpy()
            on = np.ones_like(par, bool) if parity < 0 else par == parity
            assert (np.abs(got - psi)[:, on] <= 1.5 * eps * big[:, on]).all()
            if not host:  # (a host copy comes back whole, with the staging area's other sites)
                assert (got[:, ~on] == 7.0).all()


@pytest.mark.parametrize("recon", [12, 18])
def test_gauge_load_sources(lq, recon):
    """Links from the host, the device, and a device buffer that starts at an
    odd double: the same fields in every precision."""
    import torch
    dims = (4, 6, 2, 10)  # 24 sites a parity and slice, blocks of 32
    U = synth.gauge_field(dims, "smooth", 45, eps=0.5)
    psi = on_device(synth.gaussian_spinor(dims, 46))
    odd = torch.empty(2 * U.size + 1, dtype=torch.float64, device="cuda")[1:]
    odd.copy_(torch.view_as_real(torch.from_numpy(U)).reshape(-1))
    assert odd.data_ptr() % 16 == 8
    outs = []
    for links in (on_device(U), odd, torch.from_numpy(U)):
        lat = lq.Lattice(dims, recon=recon)
        lat.gauge_load(links)
        fields = []
        for prec in ("f64", "f32", "f16", "bf16"):
            fin, fout = lat.new_field(prec), lat.new_field(prec)
            fout.zero_()
            lat.pack(fin, psi, 1, prec)
            lat.dslash(fout, fin, 0, prec=prec)
            fields.append(fout)
        lat.sync()
        outs.append(fields)
    for fields in outs[1:]:
        for a, b in zip(outs[0], fields):
            assert torch.equal(a, b)
    got = lat.canonical_spinor()
    lat.unpack(got, outs[0][0], 0, "f64")
    lat.sync()
    assert rel(got.cpu().numpy(), hop_ref(U, psi.cpu().numpy(), dims, 0)) < 1e-13


@pytest.mark.parametrize("channels", [(1, 1), (1, 2, 1), (1, 12, 12, 1), (1, 11, 5, 1)])
@pytest.mark.parametrize("dims,batch,recon", [((2, 2, 2, 2), 1, 12), ((4, 4, 6, 6), 3, 18), ((4, 2, 6, 10), 2, 12)])
def test_network_kernels_by_shape(lq, channels, dims, batch, recon):
    """The BF16 network's layers, adjoints and weight gradients against the
    FP32 network's, for every kernel that a shape selects (one input channel,
    one output channel, both, neither; odd channel counts) and lattices with a
    ragged last tile.  BF16 operands, and activations between layers, have unit
    roundoff 2^-9; sums are FP32: 5e-3 of the norm, as for single layers."""
    import torch
    lat = lq.Lattice(dims, precisions=("f64", "f32"), recon=recon)
    lat.gauge_load(on_device(synth.gauge_field(dims, "smooth", 51, eps=0.5)))
    rng = np.random.default_rng(52)
    nets = [lq.Net(lat, channels, bf16=bf, max_batch=batch) for bf in (True, False)]
    w = (rng.standard_normal(nets[0].num_weights) + 1j * rng.standard_normal(nets[0].num_weights)).astype(np.complex64)
    for n in nets:
        n.set_weights(w)

    def act(ch):
        shape = (batch, dims[3], dims[2], dims[1], dims[0], ch, 4, 3)
        return on_device((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64))

    at = 0
    for l, (cin, cout) in enumerate(zip(channels, channels[1:])):
        x, g = act(cin), act(cout)
        size = 9 * 16 * cin * cout
        res = []
        for n in nets:
            y, z = torch.empty_like(g), torch.empty_like(x)
            n.layer_apply(l, y, x, batch)
            n.layer_apply(l, z, g, batch, adjoint=True)
            n.layer_wgrad(l, x, g, batch)
            lat.sync()
            res.append((y.cpu().numpy(), z.cpu().numpy(), n.get_weights(grad=True)[1][at:at + size].numpy()))
        for got, want in zip(*res):
            assert rel(got, want) < 5e-3, (l, cin, cout)
        at += size


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 10, 2), (8, 6, 4, 10)])
@pytest.mark.parametrize("nkrylov,steps", [(1, 3), (4, 4), (5, 5), (9, 9), (24, 24), (4, 9)])
def test_fgcr_steps(lq, dims, nkrylov, steps):
    """The residual after a number of FGCR(nkrylov) steps against the smallest
    one over each cycle's Krylov space (the dots run in chunks of four vectors
    per parity).  The directions are FP32, each off by some 1e-7; 1e-5 of |b|
    covers 24 of them."""
    U = synth.gauge_field(dims, "smooth", 31, eps=0.5)
    A = oracle.clover(U, 0.12, 1.0)
    b = synth.gaussian_spinor(dims, 32)
    r, left = b.reshape(-1), steps
    while left:  # a cycle: min |r - M K y|, K = (r, M r, ..), by orthonormal vectors
        n = min(left, nkrylov)
        Q = np.zeros((n, r.size), complex)
        v = r
        for k in range(n):
            v = oracle.wilson_clover(U, A, 0.12, v.reshape(b.shape)).reshape(-1)
            for _ in range(2):
                v = v - Q[:k].T @ (Q[:k].conj() @ v)
            v = v / np.linalg.norm(v)
            Q[k] = v
        r = r - Q.T @ (Q.conj() @ r)
        left -= n
    want = np.linalg.norm(r) / np.linalg.norm(b)
    lat = lq.Lattice(dims, precisions=("f64", "f32"), gcr_nkrylov=24)
    lat.gauge_load(on_device(U))
    lat.clover_compute(0.12, 1.0)
    x = lat.canonical_spinor()
    _, st = lat.solve(x, on_device(b), 1e-30, solver=lq.SOLVER_FGCR, inner_prec="f32", nkrylov=nkrylov,
                      maxiter=steps, raise_on_error=False)
    assert st["iterations"] <= steps
    got = oracle.true_residual(U, A, 0.12, b, x.cpu().numpy())
    if st["iterations"] == steps:
        assert abs(got - want) <= 1e-5
    else:  # a cycle ended early at FP32's resolution, and so did the exact one
        assert got <= want + 1e-5


@pytest.mark.parametrize("kappa,steps", [(0.12, 8), (0.2, 5), (0.2, 8), (0.5, 2), (0.5, 12)])
def test_fgcr_second_passes(lq, kappa, steps):
    """At large kappa most of w_k lies in the span of the earlier w_j, and the
    device asks for a second Gram-Schmidt pass: as many of them, counted by
    their two launches each, as directions whose orthogonal part the exact
    recursion finds below half of |w_k|^2; and the residual of that recursion
    (FP32 directions, 1e-5 of |b| as for the steps above)."""
    dims = (4, 4, 4, 4)
    U = synth.gauge_field(dims, "smooth", 31, eps=0.5)
    A = oracle.clover(U, kappa, 0.0)
    b = synth.gaussian_spinor(dims, 32)
    r, Q, part = b.reshape(-1), [], []
    for k in range(steps):
        w = oracle.wilson_clover(U, A, kappa, r.reshape(b.shape)).reshape(-1)
        ww = np.vdot(w, w).real
        for _ in range(2):
            for q in Q:
                w = w - q * np.vdot(q, w)
        part.append(np.vdot(w, w).real / ww)
        Q.append(w / np.linalg.norm(w))
        r = r - Q[-1] * np.vdot(Q[-1], r)
    part = np.array(part)
    assert np.abs(part - 0.5).min() > 0.05  # on one side or the other beyond FP32's doubt
    lat = lq.Lattice(dims, precisions=("f64", "f32"), gcr_nkrylov=24)
    lat.gauge_load(on_device(U))
    lat.clover_compute(kappa, 0.0)
    launches = []
    for n in (1, steps):  # within one cycle; a further direction: identity, operator (2), one or two passes (2 each)
        x = lat.canonical_spinor()
        _, st = lat.solve(x, on_device(b), 1e-30, solver=lq.SOLVER_FGCR, inner_prec="f32", nkrylov=24, maxiter=n,
                          raise_on_error=False)
        assert st["iterations"] == n and st["restarts"] == 1
        launches.append(st["kernel_launches"])
    assert launches[1] - launches[0] - 5 * (steps - 1) == 2 * np.sum(part < 0.5)
    want = np.linalg.norm(r) / np.linalg.norm(b)
    assert abs(oracle.true_residual(U, A, kappa, b, x.cpu().numpy()) - want) <= 1e-5


def test_fgcr_ends_a_cycle_without_a_dependent_direction(lq):
    """A preconditioner of rank two (spins 0 and 1 alone) on constant spinors,
    which M = 1 - 8 kappa keeps: the third direction lies in the span of the
    first two.  The cycle ends with those, the next one takes the identity (the
    residual has not halved) and solves."""
    import torch
    dims, kappa = (4, 4, 4, 4), 0.1
    lat = lq.Lattice(dims, t_antiperiodic=0, precisions=("f64", "f32"), gcr_nkrylov=20)
    U = np.zeros((4, 4, 4, 4, 4, 3, 3), dtype=complex)
    U[...] = np.eye(3)
    lat.gauge_load(on_device(U))
    lat.clover_compute(kappa, 0.0)
    net = lq.Net(lat, (1, 1), bf16=False)
    W = np.zeros((9, 4, 4), complex)
    W[0] = np.diag([1.0, 0.3, 0.0, 0.0])
    net.set_weights(W.reshape(-1).astype(np.complex64))
    net.use_as_preconditioner()
    b = np.zeros((4, 4, 4, 4, 4, 3), complex)
    b[..., 0] = [0.7 + 0.2j, 0.9 - 0.4j, 1.1 + 0.3j, -0.8 + 0.6j]
    x = lat.canonical_spinor()
    _, st = lat.solve(x, on_device(b), 1e-10, solver=lq.SOLVER_FGCR, inner_prec="f32", nkrylov=20, maxiter=12)
    # without the early end the first cycle would go on to maxiter
    assert st["preconditioner_fallback"] == 1 and 2 <= st["restarts"] and 3 <= st["iterations"] < 12
    assert rel(x.cpu().numpy(), b / (1.0 - 8.0 * kappa)) < 1e-9
    net.use_as_preconditioner(False)


@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "f16spinors"])
def test_hop_right_behind_a_load(lq, prec):
    """Links loaded from the device and a hop on them, time after time with
    another field and without a wait between: the hop of a settled context,
    bit for bit (a wide and a gathering launch)."""
    import torch
    for dims in ((4, 4, 4, 6), (16, 16, 16, 16)):
        links = [on_device(synth.gauge_field(dims, "smooth", 41 + k, eps=0.5)) for k in range(2)]
        psi = on_device(synth.gaussian_spinor(dims, 43))
        lat = lq.Lattice(dims, precisions=("f64", "f32", prec))
        fin = lat.new_field(prec)
        lat.pack(fin, psi, 1, prec)
        want = []
        for u in links:
            want.append(torch.zeros_like(fin))
            lat.gauge_load(u)
            lat.sync()
            for _ in range(2):
                lat.dslash(want[-1], fin, 0, prec=prec)
            lat.sync()
        assert not torch.equal(*want)
        got = [torch.zeros_like(fin) for _ in range(40)]
        for k, f in enumerate(got):
            lat.gauge_load(links[k % 2])
            lat.dslash(f, fin, 0, prec=prec)
        lat.sync()
        for k, f in enumerate(got):
            assert torch.equal(f, want[k % 2]), (dims, k)
