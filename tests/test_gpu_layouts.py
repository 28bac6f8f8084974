"""Canonical buffers on and off a 16-byte boundary (the two forms of the layout
conversion) give the same bits, in half and full-lattice vectors, on lattices
whose last 32-site block is ragged or mostly empty."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1709_08785_gb300 import inputs

pytestmark = pytest.mark.gpu


def shifted(t):
    """A copy of t on an 8-byte but no 16-byte boundary (one complex64 or one
    double into its allocation), as (keeper, address, copy back)."""
    flat = torch.view_as_real(t).reshape(-1)
    off = 8 // flat.element_size()
    buf = torch.empty(flat.numel() + off, dtype=flat.dtype, device=t.device)
    v = buf[off:]
    v.copy_(flat)
    assert v.data_ptr() % 16 == 8
    return v, ctypes.c_void_p(v.data_ptr()), lambda: torch.view_as_complex(v.clone().view(*t.shape, 2))


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 10), (6, 4, 4, 6)])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_alignment(dims, prec, nrhs):
    from paper_1709_08785_gb300 import qcd

    ctx = qcd.Context(dims, -1)
    ctx.gauge_load(torch.from_numpy(inputs.random_gauge(dims, 0.3, 310)).cuda())
    ctx.clover_build(0.12, 1.0)
    lib, h = ctx.lib, ctx._h
    V = inputs.volume(dims)
    dt = torch.complex128 if prec in (0, 3) else torch.complex64
    v = torch.from_numpy(np.stack([inputs.gaussian_source(dims, 311 + k)[: V // 2] for k in range(nrhs)])).to(dt).cuda()
    calls = {
        "dslash": lambda o, i: lib.qcd_dslash_eo(h, o, i, 1, 1, prec, nrhs),
        "mult": lambda o, i: lib.qcd_mult_eo(h, o, i, 0, 0, prec, nrhs),
        "dhat": lambda o, i: lib.qcd_dhat(h, o, i, prec, nrhs),
        "schur": lambda o, i: lib.qcd_schur_ee(h, o, i, prec, nrhs),
        "clover": lambda o, i: lib.qcd_clover_apply(h, o, i, 0, 1, prec, nrhs),
    }
    if nrhs == 1 and prec in (0, 1):
        calls["noalloc"] = lambda o, i: lib.qcd_dslash_eo_noalloc(h, o, i, 1, 1, prec)
    for name, call in calls.items():
        out = torch.zeros_like(v)
        assert call(ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(v.data_ptr())) == 0
        keep_i, vi, _ = shifted(v)
        keep_o, vo, back = shifted(torch.zeros_like(v))
        assert call(vo, vi) == 0
        torch.cuda.synchronize()
        assert torch.equal(back(), out), name
        assert bool(torch.isfinite(torch.view_as_real(out)).all()) and float(out.abs().max()) > 0, name
    if prec == 0 and nrhs == 1:  # full vectors, both parities
        b = torch.from_numpy(inputs.gaussian_source(dims, 320)).cuda()
        x = torch.zeros_like(b)
        ctx.dirac(x, b)
        keep_i, bi, _ = shifted(b)
        keep_o, xo, back = shifted(torch.zeros_like(b))
        assert lib.qcd_dirac(h, xo, bi) == 0
        torch.cuda.synchronize()
        assert torch.equal(back(), x) and bool(torch.isfinite(torch.view_as_real(x)).all())
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_in_place(prec, nrhs):
    """out = in gives the same bits as two buffers."""
    from paper_1709_08785_gb300 import qcd

    dims = (6, 2, 4, 10)
    ctx = qcd.Context(dims, -1)
    ctx.gauge_load(torch.from_numpy(inputs.random_gauge(dims, 0.3, 310)).cuda())
    ctx.clover_build(0.12, 1.0)
    V = inputs.volume(dims)
    dt = torch.complex128 if prec in (0, 3) else torch.complex64
    v = torch.from_numpy(np.stack([inputs.gaussian_source(dims, 311 + k)[: V // 2] for k in range(nrhs)])).to(dt).cuda()
    for op in (lambda o, i: ctx.mult_eo(o, i, 0, prec=prec, nrhs=nrhs), lambda o, i: ctx.dhat(o, i, prec, nrhs),
               lambda o, i: ctx.schur_ee(o, i, prec, nrhs)):
        out, w = torch.zeros_like(v), v.clone()
        op(out, v)
        op(w, w)
        assert torch.equal(w, out)
    ctx.close()
