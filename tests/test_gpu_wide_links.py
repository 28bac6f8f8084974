"""Links that the fixed-point operators do not take (larger than SU(3), smeared
without projection, or SU(3) with an entry of zero): the FP64 and float-pair
kernels through every entry point that runs them -- operators with dagger and
several right-hand sides, solves at each level and outer arithmetic, lockstep and
batched solves, the adjoint solve -- and contexts that change between the two
kinds of field.  The FP32 and FP16 levels hold two columns of a link and take it to
be SU(3), so their solves run on a field with one unit link in it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1709_08785_gb300 import inputs

pytestmark = pytest.mark.gpu

DIMS, TBC = (6, 2, 4, 10), -1  # Vh = 240: ragged blocks
TOL = {0: 1e-13, 3: 1e-13}


def links(kind, dims, seed):
    """SU(3) but for one unit link; 1.3 SU(3); or sums of two SU(3) links, as a
    smearing step leaves them."""
    U = inputs.random_gauge(dims, 0.25, seed)
    if kind == "unit":
        U[1, 2] = np.eye(3)
        return U
    if kind == "large":
        return 1.3 * U
    return 0.7 * U + 0.3 * inputs.random_gauge(dims, 0.9, seed + 1)


def problem(kind, dims=DIMS, seed=500):
    """kappa and csw that leave D as far from singular as SU(3) links at 0.12, 1.0"""
    from paper_1709_08785_gb300 import qcd

    U = links(kind, dims, seed)
    kappa, csw = (0.12 / 1.3, 0.4) if kind == "large" else (0.12, 1.0)
    ctx = qcd.Context(dims, TBC)
    ctx.gauge_load(torch.from_numpy(U).cuda())
    ctx.clover_build(kappa, csw)
    F = oracle.clover_field(dims, U, kappa, csw)
    return dict(dims=dims, t_bc=TBC, kappa=kappa, csw=csw, U=U, F=F, ctx=ctx, b=inputs.gaussian_source(dims, seed + 2))


@pytest.fixture(scope="module", params=["unit", "large", "smeared"])
def wide(request):
    p = problem(request.param)
    p["Fi"] = oracle.invert_sites(p["F"])
    yield p
    p["ctx"].close()


@pytest.fixture(scope="module")
def su3():
    p = problem("unit", seed=504)
    yield p
    p["ctx"].close()


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def true_res(P, x, b=None):
    return oracle.true_residual(P["dims"], P["t_bc"], P["U"], P["F"], P["kappa"], P["b"] if b is None else b, x)


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_operators(wide, prec, nrhs):
    P = wide
    Vh = inputs.volume(P["dims"]) // 2
    vs = np.stack([inputs.gaussian_source(P["dims"], 510 + k)[:Vh] for k in range(nrhs)])
    inp = torch.from_numpy(vs).cuda()

    def check(call, want):
        out = torch.zeros_like(inp)
        call(out)
        got = out.cpu().numpy()
        for k in range(nrhs):
            assert rel(got[k], want(vs[k])) < TOL[prec]

    ctx, dims, t_bc, U, F, Fi, kappa = (P[k] for k in ("ctx", "dims", "t_bc", "U", "F", "Fi", "kappa"))
    for par in (0, 1):
        for dag in (False, True):
            check(lambda o: ctx.dslash_eo(o, inp, par, dag, prec, nrhs),
                  lambda v: oracle.hop_eo(dims, t_bc, U, par, v, dag))
            # F_pp^-1 H in both directions
            check(lambda o: ctx.mult_eo(o, inp, par, dag, prec, nrhs),
                  lambda v: oracle.site_apply(oracle.field_to_half(dims, par, Fi),
                                              oracle.hop_eo(dims, t_bc, U, par, v, dag)))
        check(lambda o: ctx.clover_apply(o, inp, par, True, prec, nrhs),
              lambda v: oracle.site_apply(oracle.field_to_half(dims, par, Fi), v))
    check(lambda o: ctx.dhat(o, inp, prec, nrhs), lambda v: oracle.dhat(dims, t_bc, U, Fi, kappa, v))
    check(lambda o: ctx.schur_ee(o, inp, prec, nrhs), lambda v: oracle.schur_ee(dims, t_bc, U, F, Fi, kappa, v))


def solve(P, **kw):
    bd = torch.from_numpy(P["b"]).cuda()
    x = torch.zeros_like(bd)
    info = P["ctx"].solve(bd, x, tol=1e-12, **kw)
    torch.cuda.synchronize()
    return x.cpu().numpy(), info


def check_solve(P, kw):
    x, info = solve(P, **kw)
    assert info["status"] == 0, info
    r = true_res(P, x)
    assert r <= 1e-12, (r, info)
    assert abs(info["true_resid"] - r) <= 5e-15, (info["true_resid"], r)


@pytest.mark.parametrize("kw", [dict(even_odd=0), dict(), dict(eo_hermitian=1)], ids=str)
def test_fp64_solves(wide, kw):
    check_solve(wide, dict(precision_levels=1, **kw))


@pytest.mark.parametrize("levels", [2, 3])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("herm", [0, 1])
def test_nested_solves(su3, levels, mode, herm):
    check_solve(su3, dict(precision_levels=levels, outer_df64=mode, eo_hermitian=herm))


def test_adjoint_solve(su3):
    """lam = D^-dag g: gamma5 lam solves D y = gamma5 g."""
    P = su3
    g = torch.from_numpy(P["b"]).cuda()
    lam = torch.zeros_like(g)
    info = P["ctx"].solve_adjoint(g, lam, tol=1e-12)
    assert info["status"] == 0
    five = lambda v: -np.concatenate([v[:, 2:], v[:, :2]], axis=1)  # noqa: E731
    assert true_res(P, five(lam.cpu().numpy()), five(P["b"])) <= 1e-12


@pytest.mark.parametrize("outer_df64", [0, 1])
def test_lockstep_equals_single_solves(su3, outer_df64):
    P = su3
    B = np.stack([inputs.gaussian_source(P["dims"], 520 + k) for k in range(3)])
    Bd = torch.from_numpy(B).cuda()
    X = torch.zeros_like(Bd)
    infos = P["ctx"].solve_multi(Bd, X, tol=1e-12, outer_df64=outer_df64)
    for k in range(3):
        assert infos[k]["status"] == 0
        x1 = torch.zeros_like(Bd[k])
        P["ctx"].solve(Bd[k], x1, tol=1e-12, precision_levels=2, outer_df64=outer_df64)
        assert torch.equal(X[k], x1), k
        assert true_res(P, X[k].cpu().numpy(), B[k]) <= 1e-12


@pytest.mark.parametrize("outer_df64", [0, 1, 2])
def test_batch_of_both_kinds_of_field(outer_df64):
    """Fields in fixed point and others side by side in one batch."""
    from paper_1709_08785_gb300 import qcd

    probs = [problem("unit", (4, 4, 4, 8), 530), problem("unit", DIMS, 533), problem("unit", (8, 8, 8, 8), 536)]
    for dims, seed in (((4, 4, 4, 4), 540), ((8, 4, 4, 8), 541)):
        U = inputs.random_gauge(dims, 0.25, seed)
        ctx = qcd.Context(dims, TBC)
        ctx.gauge_load(torch.from_numpy(U).cuda())
        ctx.clover_build(0.12, 1.0)
        probs.insert(1, dict(dims=dims, t_bc=TBC, kappa=0.12, U=U, F=oracle.clover_field(dims, U, 0.12, 1.0), ctx=ctx,
                             b=inputs.gaussian_source(dims, seed + 10)))
    bs = [torch.from_numpy(p["b"]).cuda() for p in probs]
    xs = [torch.zeros_like(b) for b in bs]
    infos = qcd.solve_batched([p["ctx"] for p in probs], bs, xs, [1e-10] * len(probs), precision_levels=2,
                              outer_df64=outer_df64)
    for p, x, info in zip(probs, xs, infos):
        assert info["status"] == 0 and info["restarts"] == 0, info
        r = true_res(p, x.cpu().numpy())
        assert r <= 1e-10, (p["dims"], r)
        assert abs(r - info["true_resid"]) <= 1e-12 + 0.1 * r
        p["ctx"].close()


@pytest.mark.parametrize("tuned", [False, True])
def test_a_context_changes_between_the_kinds(tuned):
    """SU(3) links, then large ones, then SU(3) again in one context: operators
    and a solve each time, with launch shapes tuned for the first field."""
    from paper_1709_08785_gb300 import qcd

    dims = DIMS
    Vh = inputs.volume(dims) // 2
    v = inputs.gaussian_source(dims, 550)[:Vh]
    b = inputs.gaussian_source(dims, 551)
    inp, bd = torch.from_numpy(v).cuda(), torch.from_numpy(b).cuda()
    ctx = qcd.Context(dims, TBC)
    U0 = inputs.random_gauge(dims, 0.25, 552)
    for scale, kappa, csw in ((1.0, 0.12, 1.0), (1.3, 0.12 / 1.3, 0.4), (1.0, 0.12, 1.0)):
        U = scale * U0
        ctx.gauge_load(torch.from_numpy(U).cuda())
        ctx.clover_build(kappa, csw)
        if tuned and scale == 1.0:
            ctx.autotune()
        F = oracle.clover_field(dims, U, kappa, csw)
        Fi = oracle.invert_sites(F)
        out = torch.zeros_like(inp)
        for prec in (0, 3):
            ctx.dhat(out, inp, prec)
            assert rel(out.cpu().numpy(), oracle.dhat(dims, TBC, U, Fi, kappa, v)) < 1e-13
            ctx.clover_apply(out, inp, 1, False, prec)
            assert rel(out.cpu().numpy(), oracle.site_apply(oracle.field_to_half(dims, 1, F), v)) < 1e-13
        for levels in (1, 2) if scale == 1.0 else (1,):
            x = torch.zeros_like(bd)
            info = ctx.solve(bd, x, tol=1e-12, precision_levels=levels)
            assert info["status"] == 0
            assert oracle.true_residual(dims, TBC, U, F, kappa, b, x.cpu().numpy()) <= 1e-12
    ctx.close()
