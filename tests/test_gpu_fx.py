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


# ---- links that fixed point is not for: each number keeps FP64's own precision ----------------------


def decoupled_links(kind, dims):
    """Links that do not mix colour 2 with the others ("blocks"), or no colours at all."""
    V = synth.volume(dims)
    rng = np.random.default_rng(31)
    U = np.zeros((4, V, 3, 3), complex)
    if kind == "unit":
        U[:] = np.eye(3)
    elif kind == "diagonal":
        U[..., range(3), range(3)] = np.exp(1j * rng.uniform(-np.pi, np.pi, (4, V, 3)))
    else:
        A = rng.standard_normal((4, V, 2, 2)) + 1j * rng.standard_normal((4, V, 2, 2))
        U[..., :2, :2] = np.linalg.qr(A)[0]
        U[..., 2, 2] = np.exp(1j * rng.uniform(-np.pi, np.pi, (4, V)))
    return U.reshape((4,) + synth.site_shape(dims) + (3, 3))


@pytest.mark.parametrize("op", ["sign", "overlap", "derivative"])
@pytest.mark.parametrize("kind", ["unit", "diagonal", "blocks"])
@pytest.mark.parametrize("dims", [(4, 3, 2, 5), (8, 8, 8, 16)])
def test_colours_that_do_not_mix_keep_their_own_precision(P, dims, kind, op):
    """Colour 2 at 1e-18 of the others gives what it gives alone, to the last bit: the others enter it only
    through links that are zero."""
    import torch

    ctx = P.Context(P.Params(dims=dims, bc=(0, 0, 0, 1), m0=M0, eps=0.1, poly_degree=4, max_nrhs=2))
    ctx.set_gauge(dev(decoupled_links(kind, dims)))
    if op == "derivative":
        P.deflate(ctx, None, [], phase=0.3)
    x = np.repeat(synth.gaussian_spinor(dims, 1, 32), 2, axis=0)
    x[..., 2] *= 1e-18
    x[1, ..., :2] = 0.0
    xd = dev(x)
    y = torch.empty_like(xd)
    if op == "sign":
        P.apply_sign_Hw(ctx, xd, y)
    elif op == "overlap":
        P.apply_overlap(ctx, xd, y, mass=0.1)
    else:
        P.apply_dDdphi(ctx, xd, y, 0.1, phase=[0.3, 0.3])
    ctx.close()
    y = y.cpu().numpy()
    assert np.abs(y[1, ..., 2]).max() > 0.0
    assert np.array_equal(y[0, ..., 2], y[1, ..., 2])


def test_links_of_very_different_sizes(P):
    """Half of the lattice with links 2^-40 times the other's, m0 = -4 (no term without a link): the derivative
    in that half, dH/dphi P(Q^2) x / h up to terms 2^-80 of it, is as accurate relative to its own size as with
    equal links."""
    import torch

    from oracle import derivative

    dims, bc, degree, hw, phase = (3, 4, 2, 14), (0, 0, 0, 2), 1, 4.0, 0.3
    U = synth.random_su3_field(dims, 0.3, seed=33)
    U[:, 7:] *= 2.0**-40
    x = synth.gaussian_spinor(dims, 1, 34)
    x[:, :11] = 0.0  # 2 n + 1 = 3 hops from the other half
    ctx = P.Context(P.Params(dims=dims, bc=bc, m0=-4.0, hw_norm=hw, eps=0.02, poly_degree=degree, max_nrhs=1))
    ctx.set_gauge(dev(U))
    P.deflate(ctx, None, [], phase=phase)
    xd = dev(x)
    y = torch.empty_like(xd)
    P.apply_dDdphi(ctx, xd, y, 0.0, phase=[phase])
    ctx.close()
    p = ov.OverlapParams(m0=-4.0, hw_norm=hw, eps=0.02, degree=degree, bc=(1.0, 1.0, 1.0, 0.0))
    px = ov.apply_poly_Q2(U, x[0], p, phase)
    want = derivative.dhw_dphi(U, px, p.bc, phase) / hw
    want[..., 2:, :] *= -1  # gamma5
    assert np.linalg.norm(want) > 0.0
    assert np.linalg.norm(y.cpu().numpy()[0] - want) <= bound(degree) * np.linalg.norm(want)


def test_a_nan_in_one_link(P):
    """It reaches the sites within 2 n + 1 hops, zeros included, and no others; in a link that no hop uses it
    reaches none."""
    dims, bc, degree = (4, 4, 2, 14), (0, 0, 0, 2), 1
    U = synth.random_su3_field(dims, 0.3, seed=35)
    x = synth.gaussian_spinor(dims, 1, 36)
    x[0, :3] = 0.0
    bad = U.copy()
    bad[0, 0, 0, 0, 0, 1, 1] = np.nan  # the x link of the first site
    y, hw = run(P, dims, bc, bad, x, degree, [0.0])
    want = oracle_sign(U, x[0], bc, hw, degree, 0.0)
    assert np.isnan(y[0, 0, 0, 0, :2]).any()
    assert np.linalg.norm(y[0, 4:] - want[4:]) <= bound(degree) * np.linalg.norm(want[4:])
    bad = U.copy()
    bad[3, -1] = np.nan  # the time links across the Dirichlet face
    y, hw = run(P, dims, bc, bad, x, degree, [0.0])
    assert np.linalg.norm(y[0] - want) <= bound(degree) * np.linalg.norm(want)


@pytest.mark.parametrize("spread, fixed", [(0.2, True), (0.4, True), (0.02, False)])
def test_which_fields_take_fixed_point(P, spread, fixed):
    """The recurrence's bytes a site tell: 196 of a fixed-point vector, 192 of an FP64 one (two applications,
    links of 576, seven vectors but for the first)."""
    import torch

    dims, degree = (6, 6, 6, 8), 4
    U = synth.random_su3_field(dims, spread, seed=37)
    x = synth.gaussian_spinor(dims, 1, 38)
    ctx = P.Context(P.Params(dims=dims, bc=(0, 0, 0, 1), m0=M0, eps=0.02, poly_degree=degree, max_nrhs=1))
    ctx.set_gauge(dev(U))
    ctx.set_profiling(True)
    xd = dev(x)
    y = torch.empty_like(xd)
    P.apply_sign_Hw(ctx, xd, y)
    want = oracle_sign(U, x[0], (0, 0, 0, 1), ctx.hw_norm, degree, 0.0)
    vectors = 7 * degree - 1
    assert ctx.read_profile(0)["clenshaw_bytes"] == synth.volume(dims) * (2 * degree * 576 + vectors * (196 if fixed else 192))
    ctx.close()
    assert np.linalg.norm(y.cpu().numpy()[0] - want) <= bound(degree) * np.linalg.norm(want)


def test_a_nan_reaches_the_derivative_through_x_hops_only(P):
    """dH/dphi has x hops only, and the derivative's recurrence starts from zeros: three y hops from a NaN, the
    result of degree 1 is what it is without."""
    import torch

    dims = (6, 8, 2, 4)
    U = synth.random_su3_field(dims, 0.3, seed=39)
    x = synth.gaussian_spinor(dims, 1, 40)
    ctx = P.Context(P.Params(dims=dims, bc=(0, 0, 0, 1), m0=M0, eps=0.02, poly_degree=1, max_nrhs=1))
    ctx.set_gauge(dev(U))
    P.deflate(ctx, None, [], phase=0.3)
    y = []
    for value in (x[0, 1, 0, 0, 2, 0, 0], np.nan):
        x[0, 1, 0, 0, 2, 0, 0] = value
        xd = dev(x)
        yd = torch.empty_like(xd)
        P.apply_dDdphi(ctx, xd, yd, 0.0, phase=[0.3])
        y.append(yd.cpu().numpy())
    ctx.close()
    assert np.isnan(y[1][0, 1, 0, 1, 1]).all() and not np.isnan(y[0]).any()
    for far in (3, 5):
        assert np.array_equal(y[1][0, 1, 0, far, 2], y[0][0, 1, 0, far, 2])


@pytest.mark.parametrize("dims, nrhs, shapes", [((4, 4, 4, 4), 8, []), ((8, 8, 8, 8), 8, [1, 2, 4]), ((8, 8, 8, 16), 3, [1, 2]),
                                                ((8, 8, 8, 16), 1, [])])
def test_only_shapes_that_differ_are_timed(P, dims, nrhs, shapes):
    """Blocks of more than four systems do not exist, and eight lanes a site take no shape at all."""
    import re

    ctx = P.Context(P.Params(dims=dims, m0=M0, eps=0.02, poly_degree=2, max_nrhs=nrhs))
    ctx.set_gauge(dev(synth.random_su3_field(dims, 0.3, seed=41)))
    x = dev(synth.gaussian_spinor(dims, nrhs, 42))
    P.apply_sign_Hw(ctx, x, x.clone())
    assert [int(k) for k in re.findall(r"(\d+)d?t?:", ctx.tune_info)] == shapes
    ctx.close()


@pytest.mark.parametrize("coeffs, hw", [([0.0, 0.0, 0.0, 0.0, 1e-12], 6.5), ([1e-12, 0.0, 1e-12, 0.0, 0.0], 6.5),
                                        ([0.0] * 5, 6.5), ([1.0, 0.5, 0.0, -0.25, 1e-30], 6.5),
                                        ([1.0, 0.5, 0.25, 0.125, 0.0625], 1e200)])
@pytest.mark.parametrize("op", ["sign", "derivative"])
def test_the_callers_coefficients(P, coeffs, hw, op):
    """Zeros among coefficients far below 1 set no unit; an operator's scale that underflows is FP64's.  The result is
    off by the bound times the largest coefficient (and the growth of T_4 below the interval).  The derivative, whose
    exact value is not at hand, scales with its coefficients by a power of two: to the last bit, but for a coefficient
    of 1, which is added without a product in a finer unit (to the bound, n + 1 times over for the derivative's sum)."""
    import torch

    dims, bc, eps = (4, 3, 2, 5), (0, 0, 0, 1), 0.1
    U = synth.random_su3_field(dims, 0.3, seed=43)
    x = synth.gaussian_spinor(dims, 1, 44)

    def run_with(cf):
        ctx = P.Context(P.Params(dims=dims, bc=bc, m0=M0, hw_norm=hw, eps=eps, poly_degree=4, coeffs=cf, max_nrhs=1))
        ctx.set_gauge(dev(U))
        xd = dev(x)
        y = torch.empty_like(xd)
        if op == "sign":
            P.apply_sign_Hw(ctx, xd, y)
        else:
            P.deflate(ctx, None, [], phase=0.3)
            P.apply_dDdphi(ctx, xd, y, 0.0, phase=[0.3])
        ctx.close()
        return y.cpu().numpy()[0]

    y = run_with(coeffs)
    if op == "sign":
        p = ov.OverlapParams(m0=M0, hw_norm=hw, eps=eps, degree=4, coeffs=np.array(coeffs), bc=(1.0, 1.0, 1.0, -1.0))
        want = ov.sign_hw(U, x[0], p, ov.SmallSpace.empty(U.shape[1:5]), 0.0)
        growth = np.cosh(4 * np.arccosh((1 + eps) / (1 - eps)))
        assert np.linalg.norm(y - want) <= bound(4) * growth * np.abs(coeffs).max() * min(1.0, 6.5 / hw)
    else:
        scaled = run_with([c * 2.0**-100 for c in coeffs]) * 2.0**100
        tol = 5 * bound(4) if 1.0 in coeffs else 0.0
        assert np.linalg.norm(scaled - y) <= tol * np.linalg.norm(y)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_coefficients_that_are_not_finite(P, bad):
    import torch

    dims = (4, 3, 2, 5)
    ctx = P.Context(P.Params(dims=dims, m0=M0, eps=0.1, poly_degree=2, coeffs=[1.0, bad, 0.5], max_nrhs=1))
    ctx.set_gauge(dev(synth.random_su3_field(dims, 0.3, seed=45)))
    x = dev(synth.gaussian_spinor(dims, 1, 46))
    y = torch.zeros_like(x)
    P.apply_sign_Hw(ctx, x, y)
    ctx.close()
    assert not np.isfinite(y.cpu().numpy()).any()
