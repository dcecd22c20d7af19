"""Inner products and norms per right-hand side (csrc/blas.cu: dot_partial_k, blocks by the length) at lengths of
one block, a part of one, several with a remainder, and more than the most blocks take.

Tolerance: a thread's sum of at most some 100 products and the tree above it, 128 x 2^-53 times the sum of the
products' magnitudes.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, nrhs", [((2, 2, 2, 2), 3), ((5, 3, 4, 7), 2), ((8, 8, 8, 8), 5), ((7, 9, 11, 13), 1),
                                        ((24, 24, 24, 16), 1)])
@pytest.mark.parametrize("per_timeslice", [False, True])
def test_inner(dims, nrhs, per_timeslice):
    import torch

    import paper_1111_6288_gb300 as P

    a, b = (synth.gaussian_spinor(dims, nrhs, seed) for seed in (61, 62))
    ctx = P.Context(P.Params(dims=dims, m0=-1.5, eps=0.02, poly_degree=2, max_nrhs=nrhs))
    ctx.set_gauge(torch.from_numpy(synth.random_su3_field(dims, 0.3, seed=63)).cuda())
    got = P.inner(ctx, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), per_timeslice=per_timeslice)
    ctx.close()
    axes = tuple(range(2 if per_timeslice else 1, a.ndim))
    want = (a.conj() * b).sum(axis=axes)
    size = (np.abs(a) * np.abs(b)).sum(axis=axes)
    assert got.shape == want.shape
    assert np.all(np.abs(got - want) <= 128 * 2.0**-53 * size)
