"""Solves near the end of the device memory: the fixed-point forms take memory
that the solve itself may need (576 bytes a site for the links, 196 for an
encoded vector), and give way to it.  The memory is held by an ordinary
allocation that leaves so many bytes a site free; solutions as with all of the
memory free: both reach tol, and A is within 0.8 of the unit matrix."""
import gc

import numpy as np
import pytest

from inputs import lattice as L

from .gpu_util import cuda, host

pytestmark = pytest.mark.gpu

DIMS = (32, 32, 32, 32)
V = 32 ** 4
TOL = 1e-8


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


@pytest.fixture(scope="module")
def system():
    import torch
    gen = torch.Generator(device="cuda:0").manual_seed(7)
    ph = torch.rand(V, 4, dtype=torch.float64, device="cuda:0", generator=gen) * 6.2831853
    U = torch.zeros(V, 4, 3, 3, dtype=torch.complex128, device="cuda:0")   # U(1) phases: quickly made
    for c in range(3):
        U[..., c, c] = torch.polar(torch.ones_like(ph), (c + 1) * ph)
    U = U.contiguous()
    b = torch.view_as_complex(torch.randn(V * 12, 2, dtype=torch.float64, device="cuda:0", generator=gen))
    return U, b


class _Fill:
    """All device memory but `per_site` bytes a site."""

    def __init__(self, per_site):
        self.leave = int(per_site * V)

    def __enter__(self):
        import torch
        gc.collect()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        assert free > self.leave
        self.held = torch.empty(free - self.leave, dtype=torch.uint8, device="cuda:0")

    def __exit__(self, *exc):
        import torch
        torch.cuda.synchronize()
        del self.held
        torch.cuda.empty_cache()


def _bicgstab(op, b, x):
    rc, st = op.dbicgstab(b, x, None, tol=TOL, max_iter=200)
    assert rc == 0 and st[0]["converged"]


def _gmresdr(op, b, x):
    rc, st, _, _ = op.gmresdr(b, x, 4, 0, TOL, 400)
    assert rc == 0 and st["converged"]


# bytes a site: BiCGStab seven vectors of 192, GMRES-DR(4) seventeen
@pytest.mark.parametrize("solve,left", [(_bicgstab, 7 * 192 - 200), (_gmresdr, 17 * 192 + 80)])
def test_links_give_way_to_a_solve(wdl, system, solve, left):
    import torch
    U, b = system
    x, ref = torch.zeros_like(b), torch.zeros_like(b)
    op = wdl.WilsonOperator(DIMS, U, 0.1)
    solve(op, b, ref)
    op.close()
    op = wdl.WilsonOperator(DIMS, U, 0.1)
    with _Fill(left):
        solve(op, b, x)
    op.close()
    assert float((x - ref).norm() / ref.norm()) <= 20 * TOL


def test_links_are_not_made_where_a_solve_needs_the_memory(wdl, system):
    import torch
    U, b = system
    x, ref = torch.zeros_like(b), torch.zeros_like(b)
    op = wdl.WilsonOperator(DIMS, U, 0.1)
    _bicgstab(op, b, ref)
    op.close()
    with _Fill(576 + 7 * 192 + 250):
        op = wdl.WilsonOperator(DIMS, U, 0.1)
        _bicgstab(op, b, x)
        op.close()
    assert float((x - ref).norm() / ref.norm()) <= 20 * TOL
