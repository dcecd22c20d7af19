"""Single Wilson applications on the caller's arrays (csrc/dslash.cu: wilson_abi_kernel and the FP64 kernel
with eight lanes a site), at the sizes where they can go wrong: site counts that fill no warp of four sites
and no block of 128, both sides of the choice between the two kernels, several right-hand sides, every
boundary condition, field phases, D_w and H_w, and arrays that overlap.

Tolerances, relative to the largest number of the result: FP64 64 units of 2^-53 (about 24 sums of 72
products of numbers below it), FP32 2e-6 and 16-bit storage 16 units of 2^-11 / 2^-8 as for the other
Wilson tests.
"""
import numpy as np
import pytest

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu
M0 = -1.5
TOL = {0: 64 * 2.0**-53, 1: 2e-6, 2: 16 * 2.0**-11, 3: 16 * 2.0**-8}


@pytest.fixture(scope="module")
def P():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1111_6288_gb300 as P

    return P


def oracle(U, x, bc, phase, hermitian):
    f = tuple((1.0, -1.0, 0.0)[b] for b in bc)
    return (dirac.hermitian_wilson if hermitian else dirac.wilson)(U, x, M0, f, phase)


def context(P, dims, bc, U, precision, nrhs):
    import torch

    ctx = P.Context(P.Params(dims=dims, bc=bc, m0=M0, eps=0.02, poly_degree=2, precision=precision, max_nrhs=nrhs))
    ctx.set_gauge(torch.from_numpy(U).cuda())
    return ctx


@pytest.mark.parametrize("precision", [0, 1, 2, 3])
@pytest.mark.parametrize("dims, nrhs", [((2, 2, 2, 2), 1), ((3, 3, 3, 5), 3), ((4, 4, 4, 4), 2), ((13, 9, 11, 13), 1),
                                        ((5, 7, 13, 6), 4), ((16, 8, 16, 8), 1)])
@pytest.mark.parametrize("bc, phases", [((0, 0, 0, 1), None), ((2, 1, 0, 2), (0.3, 0.0, -0.2, 0.1))])
def test_wilson_matches_oracle(P, dims, nrhs, bc, phases, precision):
    import torch

    U = synth.random_su3_field(dims, 0.3, seed=21)
    x = synth.gaussian_spinor(dims, nrhs, 22)
    ctx = context(P, dims, bc, U, precision, nrhs)
    xd = torch.from_numpy(x).cuda().to(ctx.spinor_dtype())
    ph = None if phases is None else list(phases[:nrhs])
    for hermitian in (False, True):
        y = torch.empty_like(xd)
        P.apply_wilson(ctx, xd, y, phase=ph, hermitian=hermitian)
        got = y.cpu().numpy().astype(np.complex128)
        for j in range(nrhs):
            want = oracle(U, x[j], bc, ph[j] if ph else 0.0, hermitian)
            assert np.abs(got[j] - want).max() <= TOL[precision] * np.abs(want).max()
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 12, 10, 12)])
def test_overlapping_arrays(P, dims, precision):
    """Different arrays that overlap by all but one vector give what separate ones give."""
    import torch

    U = synth.random_su3_field(dims, 0.3, seed=23)
    ctx = context(P, dims, (0, 0, 0, 1), U, precision, 2)
    buf = torch.from_numpy(synth.gaussian_spinor(dims, 3, 24)).cuda().to(ctx.spinor_dtype())
    want = torch.empty_like(buf[:2])
    P.apply_wilson(ctx, buf[:2].clone(), want)
    P.apply_wilson(ctx, buf[:2], buf[1:])
    assert torch.equal(buf[1:], want)
    ctx.close()
