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
@pytest.mark.parametrize("scale", [1.0, 0.6, 0.3, 1.3])
@pytest.mark.parametrize("inverse", [False, True])
def test_clover_blocks(dims, scale, inverse):
    """F and F^-1 in FP64 for SU(3) links, smaller ones, and ones below and above
    the fixed-point range (scales 0.3 and 1.3)."""
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


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 10)])
@pytest.mark.parametrize("scale", [1.0, 1.3])
@pytest.mark.parametrize("graded", [False, True])
def test_force(dims, scale, graded):
    """The link gradient in fixed point and, for links beyond its range, in FP64;
    graded: sources falling by 2^-40 from site to site, as a propagator does."""
    kappa, csw, t_bc = 0.12, 1.3, -1
    V = inputs.volume(dims)
    U = scale * inputs.random_gauge(dims, 0.3, 303)
    x, lam = inputs.gaussian_source(dims, 304), inputs.gaussian_source(dims, 305)
    if graded:
        x = x * (2.0 ** (-40.0 * (np.arange(V) % 3)))[:, None, None]
    ctx = make_ctx(dims, U, kappa, csw, t_bc)
    G = torch.zeros(U.shape, dtype=torch.complex128, device="cuda")
    ctx.force(torch.from_numpy(U).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(lam).cuda(), G)
    torch.cuda.synchronize()
    assert rel(G.cpu().numpy(), oracle.link_grad(dims, t_bc, U, kappa, csw, x, lam)) < TOL
    ctx.close()


@pytest.mark.parametrize("scale", [1.0, 1.3, 1e-7])
def test_force_takes_the_links_it_is_given(scale):
    """The gradient at other links than the loaded ones, in range or not."""
    dims, kappa, csw, t_bc = (6, 2, 4, 10), 0.12, 1.3, -1
    U = scale * inputs.random_gauge(dims, 0.3, 310)
    x, lam = inputs.gaussian_source(dims, 304), inputs.gaussian_source(dims, 305)
    ctx = make_ctx(dims, inputs.random_gauge(dims, 0.3, 303), kappa, csw, t_bc)
    G = torch.zeros(U.shape, dtype=torch.complex128, device="cuda")
    ctx.force(torch.from_numpy(U).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(lam).cuda(), G)
    torch.cuda.synchronize()
    assert rel(G.cpu().numpy(), oracle.link_grad(dims, t_bc, U, kappa, csw, x, lam)) < TOL
    ctx.close()


@pytest.mark.parametrize("scale", [0.5, 0.3, 1e-7, 1e-30])
def test_small_links_keep_their_accuracy(scale):
    """H in FP64 where its links are small against the fixed-point unit, some of
    them zero (an open boundary)."""
    dims, t_bc = (6, 2, 4, 10), -1
    Vh = inputs.volume(dims) // 2
    U = scale * inputs.random_gauge(dims, 0.3, 311)
    U[::5] = 0.0
    v = inputs.gaussian_source(dims, 312)[:Vh]
    ctx = make_ctx(dims, U, 0.12, 0.0, t_bc)
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    ctx.dslash_eo(out, inp, 0, 0, 0)
    torch.cuda.synchronize()
    assert rel(out.cpu().numpy(), oracle.hop_eo(dims, t_bc, U, 0, v)) < 1e-13
    ctx.close()


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("scale", [1.0, 1.3])
def test_operators_on_graded_vectors(prec, scale):
    """FP64 and DF64 D^ and S_ee of vectors that fall by 2^-30 from site to site
    (each site its own exponent), zero sites among them."""
    dims, kappa, csw, t_bc = (6, 2, 4, 10), 0.12, 1.0, -1
    Vh = inputs.volume(dims) // 2
    U = scale * inputs.random_gauge(dims, 0.3, 306)
    v = inputs.gaussian_source(dims, 307)[:Vh] * (2.0 ** (-30.0 * (np.arange(Vh) % 4)))[:, None, None]
    v[::7] = 0.0
    ctx = make_ctx(dims, U, kappa, csw, t_bc)
    F = oracle.clover_field(dims, U, kappa, csw)
    Fi = oracle.invert_sites(F)
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    ctx.dhat(out, inp, prec)
    assert rel(out.cpu().numpy(), oracle.dhat(dims, t_bc, U, Fi, kappa, v)) < 1e-13
    ctx.schur_ee(out, inp, prec)
    assert rel(out.cpu().numpy(), oracle.schur_ee(dims, t_bc, U, F, Fi, kappa, v)) < 1e-13
    ctx.close()


def test_non_finite_input_gives_non_finite_output():
    dims = (4, 4, 4, 4)
    ctx = make_ctx(dims, inputs.random_gauge(dims, 0.3, 308), 0.12, 1.0)
    v = inputs.gaussian_source(dims, 309)[: inputs.volume(dims) // 2]
    for bad in (np.nan, np.inf, -np.inf):
        w = v.copy()
        w[5, 1, 2] = bad
        inp = torch.from_numpy(w).cuda()
        out = torch.zeros_like(inp)
        ctx.dhat(out, inp, 0)
        got = out.cpu().numpy()
        assert not np.isfinite(got[5]).all()  # D^ holds the input at its own site
        assert np.isfinite(got).any()         # sites out of reach keep finite values
    ctx.close()


@pytest.mark.parametrize("tiny", [1e-42, 1e-38, 2.0 ** -149, 2.0 ** -126 * (1 - 2.0 ** -30)])
def test_entries_below_the_normal_range_of_fp32(tiny):
    """FP32 copies of links and clover blocks whose entries are denormal in FP32
    (the integer conversion hands them to the FP64 instruction): rounded to a
    unit of 2^-149."""
    dims, t_bc = (4, 4, 4, 4), 1
    V = inputs.volume(dims)
    U = inputs.unit_gauge(dims)
    U[..., 0, 1] = tiny
    v = np.zeros((V // 2, 4, 3), np.complex64)
    v[:, :, 1] = 2.0 ** 120  # colour 1 only: colour 0 of H v is the tiny entry times 2^120
    ctx = make_ctx(dims, U, 0.12, 0.0, t_bc)
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    ctx.dslash_eo(out, inp, 0, False, 1)
    torch.cuda.synchronize()
    U[..., 0, 1] = np.float32(tiny)
    want = oracle.hop_eo(dims, t_bc, U, 0, v.astype(np.complex128))[:, :, 0]
    assert rel(out.cpu().numpy()[:, :, 0], want) < 1e-5
    ctx.close()
    # clover entries of about `tiny`
    U = inputs.random_gauge(dims, 0.3, 313)
    kappa, csw = 0.12, tiny
    ctx = make_ctx(dims, U, kappa, csw, t_bc)
    w = np.zeros((V // 2, 4, 3), np.complex64)
    w[:, 0, 0] = 2.0 ** 120
    inp = torch.from_numpy(w).cuda()
    ctx.clover_apply(out, inp, 0, False, 1)
    torch.cuda.synchronize()
    F = oracle.clover_field(dims, U, kappa, csw)
    want = oracle.site_apply(oracle.field_to_half(dims, 0, F), w.astype(np.complex128))
    got = out.cpu().numpy()
    for s, k in ((0, 1), (0, 2), (1, 0), (1, 1), (1, 2)):  # the components without the diagonal
        # entries of both blocks, each rounded by half a unit, times 2^120 / 2 each
        assert np.abs(got[:, s, k] - want[:, s, k]).max() <= 2.0 ** (120 - 148) + 1e-5 * np.abs(want[:, s, k]).max()
    ctx.close()
