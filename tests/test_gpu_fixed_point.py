"""The fixed-point forms of the FP64 link algebra against the oracle, where
they can go wrong: ragged and two-site lattices, exact unit links, and links
that the fixed-point forms do not take (the FP64 ones take over)."""
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


def diagonal_links(dims, d, seed):
    """Links diag(d) with random phases: colours that do not mix."""
    V = inputs.volume(dims)
    ph = np.exp(2j * np.pi * np.random.default_rng(seed).random((V, 4, 3)))
    U = np.zeros((V, 4, 3, 3), np.complex128)
    U[..., range(3), range(3)] = np.asarray(d) * ph
    return U


@pytest.mark.parametrize("d", [(1.0, 1e-12, 1.0), (1.0, 0.01, 0.7), (1.0, 1.0, 1.0)])
@pytest.mark.parametrize("prec", [0, 3])
def test_colours_that_do_not_mix(d, prec):
    """H and D^ colour by colour, where a colour is small against the others: in
    the links, or (phases only) in the vector.  All terms of a component carry the
    same small factor, so its error is a few roundings of its own size."""
    dims, t_bc, kappa = (6, 2, 4, 10), -1, 0.12
    tol = {0: 1e-14, 3: 1e-13}[prec]
    Vh = inputs.volume(dims) // 2
    U = diagonal_links(dims, d, 314)
    v = inputs.gaussian_source(dims, 315)[:Vh]
    if d[1] == 1.0:
        v = v * np.array([1.0, 2.0 ** -30, 2.0 ** -70])
    ctx = make_ctx(dims, U, kappa, 0.0, t_bc)
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    ctx.dslash_eo(out, inp, 0, 0, prec)
    got, want = out.cpu().numpy(), oracle.hop_eo(dims, t_bc, U, 0, v)
    for i in range(3):
        assert rel(got[..., i], want[..., i]) < tol, i
    Fi = oracle.invert_sites(oracle.clover_field(dims, U, kappa, 0.0))
    ctx.dhat(out, inp, prec)
    got, want = out.cpu().numpy(), oracle.dhat(dims, t_bc, U, Fi, kappa, v)
    for i in range(3):
        assert rel(got[..., i], want[..., i]) < tol, i
    ctx.close()


def test_a_large_neighbour_behind_zero_links():
    """H where a site 1e25 times larger than the others is cut off by zero links."""
    dims, t_bc = (6, 2, 4, 10), -1
    Vh = inputs.volume(dims) // 2
    U = inputs.random_gauge(dims, 0.3, 316)
    stride = np.cumprod((1,) + dims[:3])
    U[0] = 0.0
    for mu in range(4):
        U[(dims[mu] - 1) * stride[mu], mu] = 0.0  # the link into site 0
    v = inputs.gaussian_source(dims, 317)[:Vh]
    v[0] *= 1e25
    ctx = make_ctx(dims, U, 0.12, 0.0, t_bc)
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    ctx.dslash_eo(out, inp, 1, 0, 0)
    assert rel(out.cpu().numpy(), oracle.hop_eo(dims, t_bc, U, 1, v)) < 1e-14
    ctx.close()


def test_force_at_links_that_do_not_mix_colours():
    """The clover part of the gradient (csw makes the hopping part negligible)
    where it is a product of small link entries only."""
    dims, kappa, csw, t_bc = (6, 2, 4, 10), 0.12, 1e45, -1
    U = diagonal_links(dims, (1.0, 1e-12, 1.0), 318)
    U[..., range(3), range(3)] = np.abs(U[..., range(3), range(3)])  # no plaquette phase: F = 1
    x, lam = inputs.gaussian_source(dims, 319), inputs.gaussian_source(dims, 320)
    x[..., [0, 2]] = 0.0
    lam[..., [0, 2]] = 0.0
    ctx = make_ctx(dims, U, kappa, csw, t_bc)
    G = torch.zeros(U.shape, dtype=torch.complex128, device="cuda")
    ctx.force(torch.from_numpy(U).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(lam).cuda(), G)
    assert rel(G.cpu().numpy(), oracle.link_grad(dims, t_bc, U, kappa, csw, x, lam)) < TOL
    ctx.close()


@pytest.mark.parametrize("scale", [1e-300, 1e-309, 1e-314])
def test_vectors_near_and_below_the_normal_range(scale):
    """The FP64 operators keep FP64's denormal values.  Down there each of the oracle's
    products (48 a component in H, 24 in F^-1) rounds by half a unit of 2^-1074."""
    dims, kappa, csw, t_bc = (6, 2, 4, 10), 0.12, 1.0, -1
    Vh = inputs.volume(dims) // 2
    U = inputs.random_gauge(dims, 0.3, 321)
    v = scale * inputs.gaussian_source(dims, 322)[:Vh]
    ctx = make_ctx(dims, U, kappa, csw, t_bc)
    F = oracle.clover_field(dims, U, kappa, csw)
    Fi = oracle.invert_sites(F)
    inp = torch.from_numpy(v).cuda()
    out = torch.zeros_like(inp)
    big = 2.0 ** 900  # (norms of denormals would underflow)

    def close(want):
        err = np.abs(out.cpu().numpy() - want).max()
        assert err <= 100 * 2.0 ** -1074 + 1e-14 * np.abs(want * big).max() / big

    ctx.dslash_eo(out, inp, 1, 0, 0)
    close(oracle.hop_eo(dims, t_bc, U, 1, v))
    ctx.dhat(out, inp, 0)
    close(oracle.dhat(dims, t_bc, U, Fi, kappa, v))
    ctx.clover_apply(out, inp, 0, True, 0)
    close(oracle.site_apply(oracle.field_to_half(dims, 0, Fi), v))
    ctx.close()


def test_force_of_vectors_whose_products_are_denormal():
    """x and lambda of 1e-155: Y, Z and the gradient are denormal (some 2^40 units of
    2^-1074), the products behind one entry (hundreds) each rounding by half a unit."""
    dims, kappa, csw, t_bc = (6, 2, 4, 10), 0.12, 3.0, -1
    U = inputs.random_gauge(dims, 0.3, 323)
    x, lam = 1e-155 * inputs.gaussian_source(dims, 324), 1e-155 * inputs.gaussian_source(dims, 325)
    ctx = make_ctx(dims, U, kappa, csw, t_bc)
    G = torch.zeros(U.shape, dtype=torch.complex128, device="cuda")
    ctx.force(torch.from_numpy(U).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(lam).cuda(), G)
    want = oracle.link_grad(dims, t_bc, U, kappa, csw, x, lam)
    assert np.abs(want).max() > 2.0 ** 35 * 2.0 ** -1074
    assert np.abs(G.cpu().numpy() - want).max() <= 1000 * 2.0 ** -1074
    ctx.close()
