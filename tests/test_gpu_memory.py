"""Calls with a large workspace where the device has little memory left: the
force and the clover build run in less, with the same results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1709_08785_gb300 import inputs

pytestmark = pytest.mark.gpu


class Filled:
    """All but `left` bytes of the device's free memory taken."""

    def __init__(self, left):
        torch.cuda.empty_cache()
        self.left = left

    def __enter__(self):
        take = torch.cuda.mem_get_info()[0] - self.left
        self.held = torch.empty(take, dtype=torch.uint8, device="cuda")
        return self

    def __exit__(self, *a):
        del self.held
        torch.cuda.empty_cache()


def test_force_and_clover_build_in_little_memory():
    """16^3x32: the force wants 365 MB or, in FP64, 113 MB; the clover build 50 MB."""
    from paper_1709_08785_gb300 import qcd

    dims, kappa, csw = (16, 16, 16, 32), 0.12, 1.0
    U = inputs.random_gauge_torch(dims, 0.3, 700)
    x, lam = (torch.from_numpy(inputs.gaussian_source(dims, s)).cuda() for s in (701, 702))
    ctxs = [qcd.Context(dims, -1) for _ in range(2)]
    G = [torch.zeros_like(U) for _ in ctxs]
    out = [torch.zeros_like(x) for _ in ctxs]
    for c in ctxs:
        c.gauge_load(U)
    a, b = ctxs
    a.clover_build(kappa, csw)
    a.force(U, x, lam, G[0])
    torch.cuda.synchronize()
    with Filled(30 << 20):
        b.clover_build(kappa, csw)
        torch.cuda.synchronize()
    with Filled(200 << 20):
        b.force(U, x, lam, G[1])
        torch.cuda.synchronize()
    for c, o in zip(ctxs, out):
        c.dirac(o, x)
    assert torch.equal(out[0], out[1])  # the same blocks
    assert float(torch.linalg.vector_norm(G[0] - G[1]) / torch.linalg.vector_norm(G[0])) < 1e-14
    for c in ctxs:
        c.close()
