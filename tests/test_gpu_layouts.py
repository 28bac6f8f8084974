"""Canonical buffers on and off a 16-byte boundary (the two forms of the layout
conversion) give the same bits, in half and full-lattice vectors, on lattices
whose last 32-site block is ragged or mostly empty."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1709_08785_gb300 import inputs

pytestmark = pytest.mark.gpu


def shifted(t):
    """A copy of t that starts one complex number into its allocation."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 10), (6, 4, 4, 6)])
@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_alignment(dims, prec, nrhs):
    from paper_1709_08785_gb300 import qcd

    ctx = qcd.Context(dims, -1)
    ctx.gauge_load(torch.from_numpy(inputs.random_gauge(dims, 0.3, 310)).cuda())
    ctx.clover_build(0.12, 1.0)
    V = inputs.volume(dims)
    dt = torch.complex128 if prec in (0, 3) else torch.complex64
    v = torch.from_numpy(np.stack([inputs.gaussian_source(dims, 311 + k)[: V // 2] for k in range(nrhs)])).to(dt).cuda()
    out = torch.zeros_like(v)
    ctx.mult_eo(out, v, 0, prec=prec, nrhs=nrhs)
    vs, os = shifted(v), shifted(torch.zeros_like(v))
    if dt == torch.complex64:
        assert vs.data_ptr() % 16 == 8
    ctx.mult_eo(os, vs, 0, prec=prec, nrhs=nrhs)
    assert torch.equal(os, out)
    if prec == 0 and nrhs == 1:  # complex128 is always on the boundary: full vectors, both parities
        b = torch.from_numpy(inputs.gaussian_source(dims, 320)).cuda()
        x, y = torch.zeros_like(b), torch.zeros_like(b)
        ctx.dirac(x, b)
        ctx.dirac(y, shifted(b))
        assert torch.equal(x, y) and bool(torch.isfinite(torch.view_as_real(x)).all())
    ctx.close()
