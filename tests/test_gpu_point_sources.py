"""Sources on a single site.  BiCGStab's first residual is orthogonal to them
(the operator's square has no part at the site: (1 - gamma)(1 + gamma) = 0), so
<r_hat, r> is zero up to rounding, and exactly in about half of the cases.  The
solver goes on with a new shadow vector: the true residual reaches tol, beside
systems that need no restart, in every precision."""
import numpy as np
import pytest

from inputs import lattice as L

from .gpu_util import cuda, host, rel_residual

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


def _sources(dims, comps):
    rng = np.random.Generator(np.random.PCG64(41))
    v = L.volume(dims)
    b = np.zeros((6, v, 12), dtype=np.complex128)
    for r in range(5):
        b[r, (7 * r) % v, :comps] = rng.normal(size=comps) + 1j * rng.normal(size=comps)
    b[5] = L.gaussian_spinor(dims, 42).reshape(v, 12)
    return b.reshape(6, -1)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (11, 7, 5, 3), (16, 16, 16, 8)])
@pytest.mark.parametrize("comps", [1, 3, 12])
@pytest.mark.parametrize("bits,delta", [(64, 0.0), (32, 0.0), (32, 1e-3), (16, 0.0)])
def test_point_sources_converge(wdl, dims, comps, bits, delta):
    U = L.gauge_field(dims, 0.5, 43)
    op = wdl.WilsonOperator(dims, cuda(U), 0.13)
    b = _sources(dims, comps)
    X = cuda(np.zeros_like(b))
    if bits == 64:
        rc, st = op.dbicgstab(cuda(b), X, None, tol=TOL, max_iter=2000)
    else:
        op.set_mixed_storage(bits)
        op.set_mixed_restart(delta)
        rc, st = op.dbicgstab_mixed(cuda(b), X, None, tol=TOL, max_iter=2000)
    op.close()
    x = host(X)
    assert rc == 0
    for r in range(6):
        assert st[r]["converged"] and not st[r]["breakdown"]
        assert rel_residual(U, dims, 0.13, x[r], b[r]) <= 1.01 * TOL
