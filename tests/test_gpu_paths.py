"""GPU tests of the kernels' alternative paths at the sizes where they can go
wrong: remainders, wrap-around on the smallest extents, both sides of a rule."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_helpers import require_cuda

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
