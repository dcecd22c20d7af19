"""The fixed-point stencil with eight lanes a site (csrc/fx.cu: fx_split_kernel, few sites) against the one with
two (more sites): both sum the same integers, so a system alone, which takes the first, and the same system
in a batch that is too large for it have the same bits.  Site counts that fill no block of 16, every boundary
condition, field phases, the operator and its derivative, sites of many magnitudes, zeros and NaNs.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
BLOCKS = 3 * 152  # of 16 sites, the most that take eight lanes a site


def bits(v):
    """The numbers as integers, so that -0.0 is not 0.0 (NaNs as 0)."""
    import torch

    return torch.where(torch.isnan(v), torch.zeros_like(v), v).view(torch.int64)


@pytest.mark.parametrize("op", ["sign", "overlap", "derivative"])
@pytest.mark.parametrize("dims", [(2, 2, 4, 4), (3, 3, 3, 3), (5, 3, 4, 7), (4, 4, 4, 4), (8, 8, 6, 5)])
@pytest.mark.parametrize("bc, phase", [((0, 0, 0, 1), 0.0), ((1, 2, 0, 2), 0.3), ((2, 0, 1, 0), -0.2)])
def test_alone_and_in_a_batch(dims, bc, phase, op):
    import torch

    import paper_1111_6288_gb300 as P

    blocks = (int(np.prod(dims)) + 15) // 16
    nrhs = BLOCKS // blocks + 1  # too many for eight lanes a site
    x = synth.gaussian_spinor(dims, 1, 51)
    rng = np.random.default_rng(52)
    x = x * 2.0 ** rng.integers(-40, 41, x.shape[:-2])[..., None, None]
    x.reshape(-1, 12)[0] = 0
    x = np.repeat(x, 3, axis=0)
    x[1].reshape(-1, 12)[-1, 5] = np.nan
    x[2] = 0
    ctx = P.Context(P.Params(dims=dims, bc=bc, m0=-1.5, hw_norm=8.0, eps=0.1, poly_degree=6, max_nrhs=nrhs))
    ctx.set_gauge(torch.from_numpy(synth.random_su3_field(dims, 0.4, seed=53)).cuda())
    if phase:
        P.deflate(ctx, None, [], phase=phase)

    def run(v):
        xd = torch.from_numpy(np.ascontiguousarray(v)).cuda()
        y = torch.empty_like(xd)
        ph = [phase] * len(v)
        if op == "sign":
            P.apply_sign_Hw(ctx, xd, y, phase=ph)
        elif op == "overlap":
            P.apply_overlap(ctx, xd, y, mass=0.1, phase=ph)
        else:
            P.apply_dDdphi(ctx, xd, y, 0.1, phase=ph)
        return torch.view_as_real(y)

    batch = run(np.concatenate([x, np.repeat(x[:1], nrhs - 3, axis=0)]))
    for j in range(3):
        alone = run(x[j : j + 1])[0]
        assert torch.equal(torch.isnan(alone), torch.isnan(batch[j]))
        assert torch.equal(bits(alone), bits(batch[j]))
    assert torch.equal(bits(batch[0]), bits(batch[-1]))
    assert not torch.isnan(batch[0]).any()
    ctx.close()
