"""The fixed-point forms of the FP64 link algebra against the oracle, where
they can go wrong: ragged and two-site lattices, exact unit links, and links
too large for the fixed-point range (the FP64 form takes over)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1709_08785_gb300 import inputs

pytestmark = pytest.mark.gpu

# FP64 products of unitary links in another order: a few ulps of the largest entry
TOL = 1e-14


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def make_ctx(dims, U, kappa, csw, t_bc=-1):
    from paper_1709_08785_gb300 import qcd

    ctx = qcd.Context(dims, t_bc)
    ctx.gauge_load(torch.from_numpy(U).cuda())
    ctx.clover_build(kappa, csw)
    return ctx


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 10), (4, 4, 6, 8)])
@pytest.mark.parametrize("scale", [1.0, 0.3, 1.3])
@pytest.mark.parametrize("inverse", [False, True])
def test_clover_blocks(dims, scale, inverse):
    """F and F^-1 in FP64 for SU(3) links, smaller ones, and ones beyond the
    fixed-point range (scale 1.3)."""
    kappa, csw = 0.12, 1.0
    U = scale * inputs.random_gauge(dims, 0.3, 300)
    ctx = make_ctx(dims, U, kappa, csw)
    F = oracle.clover_field(dims, U, kappa, csw)
    M = oracle.invert_sites(F) if inverse else F
    Vh = inputs.volume(dims) // 2
    v = inputs.gaussian_source(dims, 301)[:Vh]
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    for par in (0, 1):
        ctx.clover_apply(out, inp, par, inverse)
        torch.cuda.synchronize()
        assert rel(out.cpu().numpy(), oracle.site_apply(oracle.field_to_half(dims, par, M), v)) < TOL
    ctx.close()


def test_unit_links_give_the_identity():
    dims = (4, 4, 4, 4)
    ctx = make_ctx(dims, inputs.unit_gauge(dims), 0.12, 1.6)
    v = inputs.gaussian_source(dims, 302)[: inputs.volume(dims) // 2]
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    for inverse in (False, True):
        ctx.clover_apply(out, inp, 0, inverse)
        torch.cuda.synchronize()
        # F = 1 exactly; the chiral rotation up +- dn and back rounds twice, each
        # time by half a unit of at most 2 max|v| (per real)
        assert np.abs(out.cpu().numpy() - v).max() <= 4 * 2.0 ** -52 * np.abs(v).max()
    ctx.close()
