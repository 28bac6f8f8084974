"""Performance cases: the calls that users of this library make, timed through
its public entry points (paper_1709_08785_gb300.qcd and .autograd).

Six kinds of call stand for the library's use:
  op       one application of an operator to canonical half vectors (MULT, the
           hopping term, D^, S_ee) in each precision, one or several right-hand sides
  config   a new gauge configuration: links in, clover term and inverse built,
           the full Dirac operator applied once (the residual check of a user's
           own solver)
  solve    one solve D x = b to a true residual, one to three precision levels
  multi    the spin-colour point sources of a propagator, solved in lockstep
  batch    many independent small lattices solved in one call
  adjoint  forward solve and gradient with respect to links and source

Lattices, couplings and tolerances are those of the repository's workloads
(4^4, 16^3x32, 24^3x48, 32^3x64 and about 48^3x96; links exp(i eps H), eps 0.15-0.35;
kappa 0.115-0.124; csw 1.0-1.6; antiperiodic time).
"""
from __future__ import annotations

import math

import torch

from paper_1709_08785_gb300 import inputs, qcd
from paper_1709_08785_gb300.autograd import clover_solve

T_BC = -1
PRECS = {"f64": qcd.F64, "f32": qcd.F32, "f16": qcd.F16, "df64": qcd.DF64}


def _dims(case) -> tuple:
    return tuple(int(d) for d in case["dims"].split("x"))


def _base(dims, eps=0.25, kappa=0.124, csw=1.6) -> dict:
    return dict(dims="x".join(map(str, dims)), eps=eps, kappa=kappa, csw=csw)


def _op(dims, op, prec, nrhs=1, dagger=False, parity=0, **kw) -> dict:
    return dict(kind="op", op=op, prec=prec, nrhs=nrhs, dagger=dagger, parity=parity, **_base(dims, **kw))


def _solve(dims, levels=2, even_odd=True, hermitian=False, tol=1e-12, inner1=1e-5, inner2=1e-2, tuned=False,
           host=False, **kw) -> dict:
    return dict(kind="solve", levels=levels, even_odd=even_odd, hermitian=hermitian, tol=tol, inner1=inner1,
                inner2=inner2, tuned=tuned, host=host, **_base(dims, **kw))


def listed() -> list:
    return [
        # the smallest call: one MULT of a user's own iteration on a test lattice; latency
        dict(name="mult_f32_8c8", **_op((8, 8, 8, 8), "mult", "f32")),
        # FP16 storage, a few right-hand sides, extents that fill no tile evenly
        dict(name="schur_f16_3rhs_ragged", **_op((18, 10, 14, 22), "schur", "f16", nrhs=3)),
        # D^ at the headline lattice: a user's own Krylov solver around it
        dict(name="dhat_f32_24c48", **_op((24, 24, 24, 48), "dhat", "f32")),
        # the 12 spin-colour columns in one MULT
        dict(name="mult_f32_12rhs_24c48", **_op((24, 24, 24, 48), "mult", "f32", nrhs=12)),
        # each new configuration of an ensemble (or step of a molecular-dynamics run)
        dict(name="config_24c48", kind="config", **_base((24, 24, 24, 48))),
        # the smallest solve: no preconditioning, FP64 throughout
        dict(name="solve_fp64_plain_4c4", **_solve((4, 4, 4, 4), levels=1, even_odd=False, eps=0.3, kappa=0.12,
                                                   csw=1.0)),
        # an ordinary solve from and to pinned host buffers
        dict(name="solve_16c32_host", **_solve((16, 16, 16, 32), host=True, eps=0.3, kappa=0.12, csw=1.0)),
        # the headline: mixed-precision solve at 24^3x48 with tuned launch shapes
        dict(name="solve_24c48", **_solve((24, 24, 24, 48), tuned=True)),
        # the largest: three precision levels with the inner tolerances tuned for 48^3x96
        dict(name="solve_3level_40c80", **_solve((40, 40, 40, 80), levels=3, inner1=1e-3, inner2=3e-2)),
        # the 12 point sources of a propagator
        dict(name="propagator_32c64", kind="multi", nrhs=12, point=True, tol=1e-12,
             **_base((32, 32, 32, 64), kappa=0.1235)),
        # 48 independent lattices between 8^4 and 20^3x40
        dict(name="batch_48", kind="batch", count=48, problems=99, tol=1e-10),
        # gradient of a loss through a solve (training of a link transformation, HMC force)
        dict(name="adjoint_16c32", kind="adjoint", levels=2, tol=1e-12, **_base((16, 16, 16, 32), eps=0.3, kappa=0.12,
                                                                               csw=1.0)),
    ]


def _draw_dims(rng, lo, hi) -> tuple:
    """Even extents >= 4 of a volume near 2^u, u uniform in [lo, hi], time
    extent one to two times the spatial ones."""
    while True:
        v = 2.0 ** rng.uniform(lo, hi)
        ratio = rng.uniform(1.0, 2.2)
        side = (v / ratio) ** 0.25
        ext = [side * math.exp(rng.uniform(-0.25, 0.25)) for _ in range(3)]
        ext.append(v / (ext[0] * ext[1] * ext[2]))
        d = tuple(max(4, 2 * round(e / 2)) for e in ext)
        if d[3] <= 96 and inputs.volume(d) <= 2.0 ** hi:
            return d


def draw(rng) -> dict:
    phys = dict(eps=round(rng.uniform(0.15, 0.35), 3), kappa=round(rng.uniform(0.115, 0.124), 4), csw=1.0)
    kind = rng.choice(["op", "op", "op", "op", "config", "solve", "solve", "solve", "solve", "multi", "batch",
                       "adjoint"])
    if kind == "op":
        op = rng.choice(["mult", "dslash", "dhat", "schur"])
        return _op(_draw_dims(rng, 10, 20), op, rng.choice(sorted(PRECS)), nrhs=rng.choice([1, 1, 1, 2, 3, 5, 12, 16]),
                   dagger=op in ("mult", "dslash") and rng.random() < 0.3, parity=rng.choice([0, 1]), **phys)
    if kind == "config":
        return dict(kind="config", **_base(_draw_dims(rng, 10, 21), **phys))
    if kind == "solve":
        levels = rng.choice([1, 2, 2, 2, 3])
        even_odd = levels > 1 or rng.random() < 0.5
        return _solve(_draw_dims(rng, 8, 21 if levels > 1 else 18), levels=levels, even_odd=even_odd,
                      hermitian=even_odd and rng.random() < 0.25, tol=rng.choice([1e-8, 1e-10, 1e-12]),
                      inner1=rng.choice([1e-5, 1e-4, 1e-3]), host=rng.random() < 0.25, **phys)
    if kind == "multi":
        n = rng.choice([2, 4, 6, 12, 16])
        return dict(kind="multi", nrhs=n, point=n == 12, tol=1e-12, **_base(_draw_dims(rng, 10, 18.5), **phys))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 32), problems=rng.randint(100, 999), tol=1e-10)
    return dict(kind="adjoint", levels=2, tol=rng.choice([1e-10, 1e-12]), **_base(_draw_dims(rng, 8, 17), **phys))


# ---------------------------------------------------------------- inputs
def _mul3(A, B):
    return (A[..., :, :, None] * B[..., None, :, :]).sum(-2)


def _links(dims, eps, gen):
    """U = reunitarised exp(i eps H), H traceless Hermitian with N(0,1)
    entries (inputs.random_gauge's fields, drawn on the GPU), [V, 4, 3, 3]."""
    V = inputs.volume(dims)
    U = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    step = 1 << 18
    for s in range(0, V, step):
        n = min(step, V - s)
        X = torch.randn((n, 4, 3, 3), dtype=torch.float64, device="cuda", generator=gen)
        Y = torch.randn((n, 4, 3, 3), dtype=torch.float64, device="cuda", generator=gen)
        up = torch.triu(torch.complex(X, Y), 1)
        H = up + up.mH
        d = torch.diagonal(X, dim1=-2, dim2=-1)
        H += torch.diag_embed(d - d.mean(-1, keepdim=True))
        A = (1j * eps) * H
        E = eye + A / 4
        for k in (3, 2, 1):  # Taylor to fourth order, the rest is left to the reunitarisation
            E = eye + _mul3(A, E) / k
        a = E[..., 0]
        a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
        b = E[..., 1]
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
        c = torch.linalg.cross(a, b, dim=-1).conj()
        U[s:s + n] = torch.stack([a, b, c], dim=-1)
    return U


def _gauss(shape, gen, dtype=torch.complex128):
    v = torch.randn(shape + (2,), dtype=torch.float64, device="cuda", generator=gen)
    return torch.view_as_complex(v).to(dtype)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _source(case, dims, gen):
    V = inputs.volume(dims)
    if case["point"]:
        b = torch.zeros((case["nrhs"], V, 4, 3), dtype=torch.complex128, device="cuda")
        site = int(torch.randint(0, V, (1,), device="cuda", generator=gen).item())
        for k in range(case["nrhs"]):
            b[k, site, k // 3, k % 3] = 1.0
        return b
    return _gauss((case["nrhs"], V, 4, 3), gen)


def _fields(case, seed) -> dict:
    """The seeded fields of a case: links U and source(s) b (shared by
    prepare and exact)."""
    gen = _generator(seed)
    if case["kind"] == "batch":
        probs = []
        for p in inputs.batch_problems(case["count"], case["problems"]):
            U = _links(p["dims"], p["eps"], gen)
            probs.append(dict(dims=p["dims"], kappa=p["kappa"], csw=p["csw"], U=U,
                              b=_gauss((inputs.volume(p["dims"]), 4, 3), gen)))
        return dict(probs=probs)
    dims = _dims(case)
    V = inputs.volume(dims)
    f = dict(dims=dims, kappa=case["kappa"], csw=case["csw"], U=_links(dims, case["eps"], gen))
    if case["kind"] == "op":
        f["b"] = _gauss((case["nrhs"], V // 2, 4, 3), gen,
                        torch.complex128 if case["prec"] in ("f64", "df64") else torch.complex64)
    elif case["kind"] == "multi":
        f["b"] = _source(case, dims, gen)
    else:
        f["b"] = _gauss((V, 4, 3), gen)
        if case["kind"] == "adjoint":
            f["g"] = _gauss((V, 4, 3), gen)
    return f


def _context(f):
    ctx = qcd.Context(f["dims"], T_BC)
    ctx.gauge_load(f["U"])
    ctx.clover_build(f["kappa"], f["csw"])
    return ctx


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    f = _fields(case, seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        s["ctxs"] = [_context(p) for p in f["probs"]]
        s["b"] = [p["b"] for p in f["probs"]]
        s["x"] = [torch.zeros_like(b) for b in s["b"]]
        return s
    s["b"] = f["b"]
    if kind == "config":  # the links are the call's input
        s["ctx"], s["U"], s["out"] = qcd.Context(f["dims"], T_BC), f["U"], torch.zeros_like(f["b"])
        return s
    if kind == "adjoint":
        s["ctx"] = qcd.Context(f["dims"], T_BC)
        s["U"] = f["U"].requires_grad_(True)
        s["b"].requires_grad_(True)
        s["g"] = f["g"]
        return s
    s["ctx"] = _context(f)
    if kind == "solve" and case["host"]:
        s["b"] = f["b"].cpu().pin_memory()
        s["x"] = torch.zeros_like(s["b"], device="cpu").pin_memory()
    else:
        s["x"] = torch.zeros_like(f["b"])
    if kind == "solve" and case["tuned"]:
        s["ctx"].autotune()
    return s


def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind == "op":
        ctx, prec, n = s["ctx"], PRECS[case["prec"]], case["nrhs"]
        if case["op"] == "mult":
            ctx.mult_eo(s["x"], s["b"], case["parity"], case["dagger"], prec, n)
        elif case["op"] == "dslash":
            ctx.dslash_eo(s["x"], s["b"], case["parity"], case["dagger"], prec, n)
        elif case["op"] == "dhat":
            ctx.dhat(s["x"], s["b"], prec, n)
        else:
            ctx.schur_ee(s["x"], s["b"], prec, n)
        return s["x"]
    if kind == "config":
        s["ctx"].gauge_load(s["U"])
        s["ctx"].clover_build(case["kappa"], case["csw"])
        s["ctx"].dirac(s["out"], s["b"])
        return s["out"]
    if kind == "solve":
        s["ctx"].solve(s["b"], s["x"], tol=case["tol"], precision_levels=case["levels"], even_odd=case["even_odd"],
                       eo_hermitian=case["hermitian"], inner_tol=[case["inner1"], case["inner2"]])
        return s["x"]
    if kind == "multi":
        s["ctx"].solve_multi(s["b"], s["x"], tol=case["tol"])
        return s["x"]
    if kind == "batch":
        qcd.solve_batched(s["ctxs"], s["b"], s["x"], [case["tol"]] * len(s["ctxs"]), precision_levels=2)
        return torch.cat([x.reshape(-1) for x in s["x"]])
    s["U"].grad = s["b"].grad = None
    x = clover_solve(s["U"], s["b"], s["ctx"], case["kappa"], case["csw"], tol=case["tol"], levels=case["levels"])
    x.backward(s["g"])
    return dict(x=x.detach(), grad_U=s["U"].grad, grad_b=s["b"].grad)


# ---------------------------------------------------------------- work
# Bytes per even site of one D^ application at a precision, every field read
# once: the links of both parities, F^-1 of both, the vector in and out
_DHAT = {"f64": 8 * 144 + 2 * 576 + 2 * 192, "f32": 8 * 48 + 2 * 288 + 2 * 96, "f16": 8 * 24 + 2 * 144 + 2 * 52}
_SP = {"f64": 192, "f32": 96, "f16": 52}
# Typical iteration counts of the fields drawn here (35 FP64 iterations to
# 1e-12 at 24^3x48; 47 FP32 inner ones in two outer ones; 38 FP16 ones)
_ITER = {1: 35, 2: 47, 3: 38}


def _solve_work(Vh, levels, tol, even_odd=True):
    prec = {1: "f64", 2: "f32", 3: "f16"}[levels]
    it = _ITER[levels] * math.log(tol) / math.log(1e-12) * (1.0 if even_odd else 2.0)
    # an iteration: two D^ (each reads a vector and writes one), then the
    # updates of s, x, r, p: ten further reads and writes of a vector
    by = it * (2 * _DHAT[prec] + 10 * _SP[prec])
    fl = it * (2 * (2 * 1824 + 48) + 6 * 96 + 6 * 48)
    if levels > 1:  # four outer D^, the source, reconstruction and residual in FP64
        by += 7 * _DHAT["f64"]
        fl += 7 * 2 * 1824
    return by * Vh, fl * Vh


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ws = [_solve_work(inputs.volume(p["dims"]) // 2, 2, case["tol"])
              for p in inputs.batch_problems(case["count"], case["problems"])]
        return {"bytes": sum(w[0] for w in ws), "flops": sum(w[1] for w in ws)}
    V = inputs.volume(_dims(case))
    Vh = V // 2
    if kind == "op":
        wide = case["prec"] in ("f64", "df64")
        p = "f64" if wide else case["prec"]
        link, clov = {"f64": (144, 576), "f32": (48, 288), "f16": (24, 144)}[p]
        two = case["op"] in ("dhat", "schur")
        fields = 8 * link + clov * ({"mult": 1, "dslash": 0, "dhat": 2, "schur": 2}[case["op"]])
        io = 2 * (192 if wide else 96) * case["nrhs"]
        fl = (1320 * (2 if two else 1) + 504 * {"mult": 1, "dslash": 0, "dhat": 2, "schur": 2}[case["op"]])
        return {"bytes": (fields + io) * Vh, "flops": fl * Vh * case["nrhs"]}
    if kind == "config":
        # links in; their copies (FP64, DF64, FP32, FP16) and F, F^-1 in four
        # precisions out; D: links, F, vector in and out.  Flops: 24 leaves
        # of two 3x3 products each (shared halves), the 6x6 inverses, D
        return {"bytes": V * (576 + 4 * (144 + 144 + 48 + 24) + 2 * (576 + 576 + 288 + 144) + 576 + 576 + 2 * 192),
                "flops": V * (24 * 2 * 198 + 2 * 2000 + 1824)}
    if kind == "solve":
        by, fl = _solve_work(Vh, case["levels"], case["tol"], case["even_odd"])
        return {"bytes": by, "flops": fl}
    if kind == "multi":
        by, fl = _solve_work(Vh, 2, case["tol"])
        n = case["nrhs"]
        # links and clover of an FP32 D^ once for all right-hand sides
        shared = _ITER[2] * 2 * (_DHAT["f32"] - 2 * 96) * Vh
        return {"bytes": n * by - (n - 1) * shared, "flops": n * fl}
    by, fl = _solve_work(Vh, 2, case["tol"])
    return {"bytes": 2 * by + V * (2 * 576 + 2 * 3200), "flops": 2 * fl + V * (24 * 2 * 198 + 2 * 2000 + 4 * 6000)}


def tolerance(case):
    kind = case["kind"]
    if kind == "op":
        # measured against exact(): FP64 2.3e-16, FP32 1.3e-7, FP16 storage
        # 3.4e-4; DF64 rounds to 2^-48 = 3.6e-15 per operation
        return {"rel": {"f64": 2e-15, "df64": 3e-14, "f32": 5e-7, "f16": 1.5e-3}[case["prec"]]}
    if kind == "config":
        return {"rel": 2e-15}
    # a solution is fixed to the residual tol times the condition number of D:
    # measured 2.3 tol (plain FP64 at 4^4) and 0.03-0.4 tol (two levels)
    return {"rel": 10.0 * case["tol"]}


# ---------------------------------------------------------------- 64-bit reference
def _gammas():
    s = torch.zeros((3, 2, 2), dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:] = -1j * s[k]
        g[k, 2:, :2] = 1j * s[k]
    g[3] = torch.diag(torch.tensor([1, 1, -1, -1], dtype=torch.complex128))
    return g.cuda()


class _Reference:
    """D = F - kappa H of the package's conventions in complex128 torch."""

    def __init__(self, dims, U, kappa, csw):
        self.dims, self.kappa = dims, kappa
        self.shape = (dims[3], dims[2], dims[1], dims[0])
        self.U = U.reshape(self.shape + (4, 3, 3))
        self.g = _gammas()
        self.eye = torch.eye(4, dtype=torch.complex128, device="cuda")
        self.csw = csw
        V = inputs.volume(dims)
        s = torch.arange(V, device="cuda")
        par, r = torch.zeros_like(s), s
        for d in dims:
            par = par + r % d
            r = r // d
        self.par = par % 2
        F6 = []
        for mu in range(4):
            for nu in range(mu + 1, 4):
                F6.append((mu, nu, self._strength(mu, nu)))
        self.F6 = F6
        self.Finv = None

    def _shift(self, f, mu, n):
        """f at the site + n mu."""
        return torch.roll(f, -n, dims=3 - mu)

    def _strength(self, mu, nu):
        A, B = self.U[..., mu, :, :], self.U[..., nu, :, :]
        sh = self._shift
        plaq = A @ sh(B, mu, 1) @ sh(A, nu, 1).mH @ B.mH
        Q = plaq
        # the other three leaves: the plaquettes at n - mu, n - mu - nu, n - nu
        # carried to n along their own links
        Q = Q + B @ sh(sh(A, nu, 1), mu, -1).mH @ sh(B, mu, -1).mH @ sh(A, mu, -1)
        Amn, Bmn = sh(sh(A, mu, -1), nu, -1), sh(sh(B, mu, -1), nu, -1)
        Q = Q + sh(A, mu, -1).mH @ Bmn.mH @ Amn @ sh(B, nu, -1)
        Q = Q + sh(B, nu, -1).mH @ sh(A, nu, -1) @ sh(sh(B, mu, 1), nu, -1) @ A.mH
        return (Q - Q.mH) / 8j

    def hop(self, v, dagger=False):
        v = v.reshape(self.shape + (4, 3))
        out = torch.zeros_like(v)
        for mu in range(4):
            Um = self.U[..., mu, :, :]
            fwd, bwd = self.eye - self.g[mu], self.eye + self.g[mu]
            if dagger:
                fwd, bwd = bwd, fwd
            sign = torch.ones((self.dims[3], 1, 1, 1, 1, 1), dtype=torch.float64, device="cuda")
            sb = sign.clone()
            if mu == 3:
                sign[-1], sb[0] = T_BC, T_BC
            # (U psi)_{a i} = sum_j U_ij psi_aj
            out = out + torch.einsum("ab,...bi->...ai", fwd, sign * (self._shift(v, mu, 1) @ Um.mT))
            out = out + torch.einsum("ab,...bi->...ai", bwd, sb * self._shift(v @ Um.conj(), mu, -1))
        return out.reshape(-1, 4, 3)

    def clover(self, v):
        v = v.reshape(self.shape + (4, 3))
        out = v.clone()
        for mu, nu, F in self.F6:
            sig = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
            out = out - self.csw * self.kappa * torch.einsum("ab,...bi->...ai", sig, v @ F.mT)
        return out.reshape(-1, 4, 3)

    def clover_inverse(self, v):
        if self.Finv is None:
            n = inputs.volume(self.dims)
            M = torch.zeros((n, 12, 12), dtype=torch.complex128, device="cuda")
            for k in range(12):
                e = torch.zeros((n, 4, 3), dtype=torch.complex128, device="cuda")
                e[:, k // 3, k % 3] = 1.0
                M[:, :, k] = self.clover(e).reshape(n, 12)
            for s in range(0, n, 1 << 16):
                M[s:s + (1 << 16)] = torch.linalg.inv(M[s:s + (1 << 16)])
            self.Finv = M
        return (self.Finv @ v.reshape(-1, 12, 1)).reshape(-1, 4, 3)

    def D(self, v):
        return self.clover(v) - self.kappa * self.hop(v)

    def embed(self, h, parity):
        v = torch.zeros((self.par.numel(), 4, 3), dtype=torch.complex128, device="cuda")
        v[self.par == parity] = h.to(torch.complex128)
        return v

    def half(self, v, parity):
        return v[self.par == parity]

    def op(self, name, h, out_parity, dagger):
        if name in ("mult", "dslash"):
            w = self.hop(self.embed(h, 1 - out_parity), dagger)
            return self.half(self.clover_inverse(w) if name == "mult" else w, out_parity)
        e = self.embed(h, 0)
        odd = self.embed(self.half(self.clover_inverse(self.hop(e)), 1), 1)
        w = self.hop(odd)
        k2 = self.kappa * self.kappa
        if name == "dhat":
            return self.half(e - k2 * self.clover_inverse(w), 0)
        return self.half(self.clover(e) - k2 * w, 0)

    def solve(self, b, apply=None, tol=3e-15):
        """BiCGStab on D to the rounding limit."""
        apply = apply or self.D
        x = torch.zeros_like(b)
        for _ in range(3):  # restarts from the true residual
            r = b - apply(x)
            rt, p = r.clone(), r.clone()
            rho = torch.vdot(rt.reshape(-1), r.reshape(-1))
            bn = float(torch.linalg.vector_norm(b))
            if float(torch.linalg.vector_norm(r)) <= tol * bn:
                break
            for _ in range(300):
                q = apply(p)
                a = rho / torch.vdot(rt.reshape(-1), q.reshape(-1))
                s = r - a * q
                t = apply(s)
                w = torch.vdot(t.reshape(-1), s.reshape(-1)) / torch.vdot(t.reshape(-1), t.reshape(-1))
                x = x + a * p + w * s
                r = s - w * t
                if float(torch.linalg.vector_norm(r)) <= 0.3 * tol * bn:
                    break
                new = torch.vdot(rt.reshape(-1), r.reshape(-1))
                p = r + (new / rho) * (a / w) * (p - w * q)
                rho = new
        return x


# Lattice sites times solves above which the reference takes too long
_EXACT_SITES = 700_000


def _sites(case) -> int:
    if case["kind"] == "batch":
        return sum(inputs.volume(p["dims"]) for p in inputs.batch_problems(case["count"], case["problems"]))
    return inputs.volume(_dims(case)) * (case["nrhs"] if case["kind"] == "multi" else 1)


def exact(case, seed):
    kind = case["kind"]
    if _sites(case) > (_EXACT_SITES if kind in ("solve", "multi", "batch", "adjoint") else 1 << 21):
        return None
    f = _fields(case, seed)
    if kind == "batch":
        out = []
        for p in f["probs"]:
            out.append(_Reference(p["dims"], p["U"], p["kappa"], p["csw"]).solve(p["b"]).reshape(-1))
        return torch.cat(out)
    R = _Reference(f["dims"], f["U"], f["kappa"], f["csw"])
    if kind == "op":
        return torch.stack([R.op(case["op"], h, case["parity"], case["dagger"]) for h in f["b"]])
    if kind == "config":
        return R.D(f["b"])
    if kind == "solve":
        return R.solve(f["b"])
    if kind == "multi":
        return torch.stack([R.solve(b) for b in f["b"]])
    x = R.solve(f["b"])
    g5 = R.g[0] @ R.g[1] @ R.g[2] @ R.g[3]
    five = lambda v: torch.einsum("ab,...bi->...ai", g5, v)  # noqa: E731
    lam = five(R.solve(five(f["g"])))  # D^-dag = gamma5 D^-1 gamma5
    # dL/dU of -Re <lam, D[U] x> with x and lam held fixed
    U = f["U"].detach().clone().requires_grad_(True)
    (-torch.vdot(lam.reshape(-1), _Reference(f["dims"], U, f["kappa"], f["csw"]).D(x).reshape(-1)).real).backward()
    return dict(x=x, grad_U=U.grad, grad_b=lam)
