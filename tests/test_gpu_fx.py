"""The fixed-point recurrences of the FP64 operators (csrc/fx.cu) against the oracle, at the sizes where
they can go wrong: site counts that fill no tile of 32 sites and no warp of 16, the smallest extents,
systems that fill no block, every boundary condition, field phases, links that are not SU(3), vectors whose
sites differ by many orders of magnitude, zeros and NaNs.

Tolerance: the library's recurrence rounds each of its 2 n + 1 applications to 2^-55 of a site's largest
number, the oracle's to a few 2^-53; with 8 units of 2^-53 per application of both, relative to the result
in the 2-norm, the bound is 8 (2 n + 1) 2^-53 times the growth of a Clenshaw recurrence, at most n + 1.
"""
import numpy as np
import pytest

import synth
from oracle import overlap as ov

pytestmark = pytest.mark.gpu
M0 = -1.5
U64 = 2.0**-53


@pytest.fixture(scope="module")
def P():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1111_6288_gb300 as P

    return P


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def bound(n):
    return 8 * (2 * n + 1) * U64 * (n + 1)


def run(P, dims, bc, U, x, degree, phases, eps=0.02, hw=None):
    import torch

    ctx = P.Context(P.Params(dims=dims, bc=bc, m0=M0, hw_norm=hw or 0.0, eps=eps, poly_degree=degree,
                             max_nrhs=len(x)))
    ctx.set_gauge(dev(U))
    for ph in set(phases):
        if ph:
            P.deflate(ctx, None, [], phase=ph)
    xd = dev(x)
    y = torch.empty_like(xd)
    P.apply_sign_Hw(ctx, xd, y, phase=phases)
    hw = ctx.hw_norm
    ctx.close()
    return y.cpu().numpy(), hw


def oracle_sign(U, x, bc, hw, degree, phase, eps=0.02):
    p = ov.OverlapParams(m0=M0, hw_norm=hw, eps=eps, degree=degree, bc=tuple((1.0, -1.0, 0.0)[b] for b in bc))
    return ov.sign_hw(U, x, p, ov.SmallSpace.empty(U.shape[1:5]), phase)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 7), (4, 4, 4, 4), (5, 3, 3, 11), (8, 2, 6, 5)])
@pytest.mark.parametrize("bc", [(0, 0, 0, 1), (2, 0, 0, 2), (1, 2, 1, 0)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_sign_matches_oracle(P, dims, bc, nrhs):
    degree = 5
    U = synth.random_su3_field(dims, 0.3, seed=11)
    x = synth.gaussian_spinor(dims, nrhs, 12)
    phases = [0.0, 0.3, -0.2][:nrhs]
    y, hw = run(P, dims, bc, U, x, degree, phases)
    for j in range(nrhs):
        want = oracle_sign(U, x[j], bc, hw, degree, phases[j])
        assert np.linalg.norm(y[j] - want) <= bound(degree) * np.linalg.norm(want)


@pytest.mark.parametrize("scale", [1e-3, 0.4, 5.0])
def test_links_that_are_not_su3(P, scale):
    """Links of any size are stored divided by a power of two."""
    dims, bc, degree = (4, 3, 2, 5), (0, 0, 0, 1), 4
    U = scale * synth.random_su3_field(dims, 0.3, seed=3)
    x = synth.gaussian_spinor(dims, 1, 4)
    hw = 2.5 + 4 * scale
    y, hw = run(P, dims, bc, U, x, degree, [0.0], hw=hw)
    want = oracle_sign(U, x[0], bc, hw, degree, 0.0)
    assert np.linalg.norm(y[0] - want) <= bound(degree) * np.linalg.norm(want)


def test_every_site_has_its_own_exponent(P):
    """Two sources more than 2 (2 n + 1) time slices apart, one 2^-200 times the other: neither reaches the
    other's sites, and each result is as accurate relative to its own size as alone."""
    dims, bc, degree = (2, 4, 2, 16), (0, 0, 0, 2), 1
    U = synth.random_su3_field(dims, 0.3, seed=5)
    x = synth.gaussian_spinor(dims, 1, 6)
    x[0, 1:8] = 0.0
    x[0, 9:] = 0.0
    x[0, 8] *= 2.0**-200
    y, hw = run(P, dims, bc, U, x, degree, [0.0])
    want = oracle_sign(U, x[0], bc, hw, degree, 0.0)
    for part in (slice(0, 4), slice(5, 12)):
        assert np.linalg.norm(want[part]) > 0.0
        assert np.linalg.norm(y[0, part] - want[part]) <= bound(degree) * np.linalg.norm(want[part])
    assert np.all(y[0, 4] == 0.0) and np.all(y[0, 12:] == 0.0)


def test_zero_and_nan(P):
    dims, bc, degree = (4, 4, 2, 12), (0, 0, 0, 2), 1
    U = synth.random_su3_field(dims, 0.3, seed=7)
    x = synth.gaussian_spinor(dims, 3, 8)
    x[0] = 0.0
    x[1, 0, 0, 0, 0, 0, 0] = np.nan
    x[2, 0, 0, 0, 0, 1, 2] = np.inf
    y, hw = run(P, dims, bc, U, x, degree, [0.0] * 3)
    assert np.all(y[0] == 0.0)
    for j in (1, 2):  # within 2 n + 1 = 3 hops of the bad site, and nowhere else
        assert np.isnan(y[j, 0, 0, 0, 0]).all()
        clean = x[j].copy()
        clean[0, 0, 0, 0] = 0.0
        want = oracle_sign(U, clean, bc, hw, degree, 0.0)
        assert np.linalg.norm(y[j, 4:] - want[4:]) <= bound(degree) * np.linalg.norm(want[4:])


@pytest.mark.parametrize("hw, eps", [(4.0, 0.875), (2.0, 0.5), (8.0, 0.96875), (4.0, 0.75)])
@pytest.mark.parametrize("degree", [1, 4])
def test_operator_coefficients_that_are_powers_of_two(P, hw, eps, degree):
    """alpha = 4 / ((1 - eps) h^2) of exactly 2 and 1: half of it, or all of it, is the coefficient of a plain
    step as well.  Only the last step of the recurrence is halved."""
    dims, bc = (4, 3, 2, 5), (0, 0, 0, 1)
    assert 4 / ((1 - eps) * hw**2) in (1.0, 2.0)
    U = synth.random_su3_field(dims, 0.3, seed=21)
    x = synth.gaussian_spinor(dims, 1, 22)
    y, _ = run(P, dims, bc, U, x, degree, [0.0], eps=eps, hw=hw)
    want = oracle_sign(U, x[0], bc, hw, degree, 0.0, eps=eps)
    # the spectrum of Q^2, [0, (6.5 / hw)^2], leaves [eps, 1] on both sides: T_n of its far ends is the growth
    ends = (1 + eps) / (1 - eps), (2 * (6.5 / hw) ** 2 - (1 + eps)) / (1 - eps)
    growth = np.cosh(degree * np.arccosh(max(ends)))
    assert np.linalg.norm(y[0] - want) <= bound(degree) * growth * np.linalg.norm(x[0])
    assert np.linalg.norm(want) > 1e3 * bound(degree) * growth * np.linalg.norm(x[0])
