"""Gram matrices and rotations of a block of vectors (csrc/blas.cu: multidot_k on the upper tiles of 8 x 8 with
their mirror images, combine_k) at block sizes around the tile's edge, through the call that
orthonormalises a caller's vectors and the projection that then uses them.

Tolerances, relative to |x|: FP64 sums of 12 V products twice over, 32 V 2^-53 x 12; FP32 vectors and
coefficients 64 x 2^-24.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 17, 32, 33, 65])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 4, 7)])
def test_orthonormalised_block_projects(dims, n, precision):
    import torch

    import paper_1111_6288_gb300 as P

    V = synth.gaussian_spinor(dims, n, 41)
    V = V + 0.5 * V[:1]  # not close to orthogonal
    x = synth.gaussian_spinor(dims, 3, 42)
    lam = np.where(np.arange(n) % 3 == 0, -0.1, 0.2)
    ctx = P.Context(P.Params(dims=dims, m0=-1.5, eps=0.02, poly_degree=2, precision=precision, max_nrhs=3))
    ctx.set_gauge(torch.from_numpy(synth.random_su3_field(dims, 0.3, seed=43)).cuda())
    P.deflate(ctx, torch.from_numpy(V).cuda(), lam)
    xd = torch.from_numpy(x).cuda().to(ctx.spinor_dtype())
    ys, xp = torch.empty_like(xd), torch.empty_like(xd)
    P.project_small(ctx, xd, ys, xp)
    ys, xp = (t.cpu().numpy().astype(np.complex128).reshape(3, -1).T for t in (ys, xp))
    ctx.close()
    Q, _ = np.linalg.qr(V.reshape(n, -1).T)
    X = x.reshape(3, -1).T
    c = Q.conj().T @ X
    tol = 12 * 32 * np.prod(dims) * 2.0**-53 if precision == 0 else 64 * 2.0**-24
    norm = np.linalg.norm(X, axis=0)
    assert np.all(np.linalg.norm(xp - (X - Q @ c), axis=0) <= tol * norm)
    assert np.all(np.linalg.norm(ys - Q @ (np.sign(lam)[:, None] * c), axis=0) <= tol * norm)
