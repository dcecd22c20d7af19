"""The rounding error of the block products (csrc/blas.cu: ProductSum) is that of sums rounded once a product.

A sum of N products of random signs, rounded once a product, is off by sqrt(N / 2) r of its size (the partial sums
grow with the square root of the terms), r = 0.212 x 2^-23 the mean square rounding of an FP32 number whose
mantissa is spread evenly over the logarithm.  V diag(s) V^+ x of N = 128 vectors adds the roundings of the FP32
copy of V and of the coefficients (r each) and those of V^+ x, below 3 r in sum.  Two roundings a product are
sqrt(2) times the first: 11.3 r against 8 r.  The bound lies between them, 9.5 r, the mean over 12 V x 4 numbers being
sure to a percent.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 2, 4])
def test_projection_rounds_once_a_product(nrhs):
    import torch

    import paper_1111_6288_gb300 as P

    dims, n = (8, 8, 8, 8), 128
    V = synth.gaussian_spinor(dims, n, 71)
    x = synth.gaussian_spinor(dims, nrhs, 72).astype(np.complex64)
    lam = np.where(np.arange(n) % 2, 1.0, -1.0)
    ctx = P.Context(P.Params(dims=dims, m0=-1.5, eps=0.02, poly_degree=2, precision=1, max_nrhs=4))
    ctx.set_gauge(torch.from_numpy(synth.random_su3_field(dims, 0.3, seed=73)).cuda())
    P.deflate(ctx, torch.from_numpy(V).cuda(), lam)
    xd = torch.from_numpy(x).cuda()
    ys, xp = torch.empty_like(xd), torch.empty_like(xd)
    P.project_small(ctx, xd, ys, xp)
    ctx.close()
    Q, R = np.linalg.qr(V.reshape(n, -1).T)
    Q = Q * (np.diag(R) / np.abs(np.diag(R)))
    want = Q @ (lam[:, None] * (Q.conj().T @ x.reshape(nrhs, -1).T.astype(np.complex128)))
    err = np.linalg.norm(ys.cpu().numpy().reshape(nrhs, -1).T - want) / np.linalg.norm(want)
    assert err <= 9.5 * 0.212 * 2.0**-23, err / (0.212 * 2.0**-23)
