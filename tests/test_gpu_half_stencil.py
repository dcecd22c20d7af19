"""The 16-bit stencil's factors (csrc/dslash.cu: site scales, boundary factors, field phases folded into the
accumulation; csrc/half_store.h: links of three rows) on vectors whose sites differ by many orders of
magnitude, so that a factor taken from another site or left out shows.

Bound, per site and component, u = 2^-11 (FP16) or 2^-8 (BF16): stored numbers and link entries are off by
at most u times the largest of their site, or of 1; a hop's half spinor is a sum of two numbers and its link
product a sum over three colours, so with complex factors a hop of a site of magnitude m is off by at most
3 (2 m u + 2 m u) sqrt(2) sqrt(2) / 2 = 12 u m, the mass term (|4 + m0| <= 3) by 3 u m, and storing the result rounds a
sum of at most 3 m + sum over hops of 6 m once more.  Together at most 18 u times the sum of the magnitudes of the
site and its neighbours; 20 u leaves room for the FP32 roundings.
"""
import numpy as np
import pytest

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu
M0 = -1.5


@pytest.mark.parametrize("precision", [2, 3])
@pytest.mark.parametrize("dims, nrhs", [((2, 2, 2, 2), 2), ((5, 3, 4, 7), 3), ((8, 4, 4, 8), 5), ((16, 8, 4, 4), 1)])
@pytest.mark.parametrize("bc, phases", [((0, 0, 0, 1), None), ((1, 2, 0, 2), (0.3, 0.0, -0.2, 0.1, 2.0))])
def test_sites_of_many_magnitudes(dims, nrhs, bc, phases, precision):
    import torch

    import paper_1111_6288_gb300 as P

    u = 2.0**-11 if precision == 2 else 2.0**-8
    U = synth.random_su3_field(dims, 0.4, seed=31)
    x = synth.gaussian_spinor(dims, nrhs, 32)
    rng = np.random.default_rng(33)
    x *= 2.0 ** rng.integers(-30, 31, x.shape[:-2])[..., None, None]
    ctx = P.Context(P.Params(dims=dims, bc=bc, m0=M0, eps=0.02, poly_degree=2, precision=precision, max_nrhs=nrhs))
    ctx.set_gauge(torch.from_numpy(U).cuda())
    xd = torch.from_numpy(x).cuda().to(ctx.spinor_dtype())
    y = torch.empty_like(xd)
    ph = None if phases is None else list(phases[:nrhs])
    P.apply_wilson(ctx, xd, y, phase=ph, hermitian=True)
    got = y.cpu().numpy().astype(np.complex128)
    ctx.close()
    f = tuple((1.0, -1.0, 0.0)[b] for b in bc)
    for j in range(nrhs):
        want = dirac.hermitian_wilson(U, x[j], M0, f, ph[j] if ph else 0.0)
        m = np.maximum(np.abs(x[j].real), np.abs(x[j].imag)).max(axis=(-2, -1))
        near = m + sum(np.roll(m, s, axis) for axis in range(4) for s in (1, -1))
        assert np.all(np.abs(got[j] - want).max(axis=(-2, -1)) <= 20 * u * near)
