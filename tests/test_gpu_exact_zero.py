"""BiCGStab's scalar steps (bicg_fin.cuh) where a dot is zero exactly.

kappa = 0 makes A the unit matrix: from x0 = 0 the first step has alpha = 1,
s = t = 0 and r = 0, every number a power of two times the source, so the
expected values hold exactly: one product counted (t = A s = 0 is none),
recursive and true residual 0, x = b.  Sizes: the scalar step in the last
block (4^4), in a kernel of its own over 640 and 1040 partials.  At 1e-150 the
squares are 1e-300: any value but zero in place of ||r||^2 shows against them.
"""
import numpy as np
import pytest

from inputs import lattice as L

from .gpu_util import cuda, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 16, 16, 10), (26, 16, 16, 10)])
@pytest.mark.parametrize("scale", [1.0, 1e-150])
@pytest.mark.parametrize("even_odd", [False, True])
def test_zero_residual_is_zero(wdl, dims, scale, even_odd):
    op = wdl.WilsonOperator(dims, cuda(L.gauge_field(dims, 0.5, 31)), 0.0)
    op.set_operator(even_odd)
    b = np.zeros((1, op.op_n), dtype=np.complex128)
    b[0, 5] = scale
    X = cuda(np.zeros_like(b))
    rc, st = op.dbicgstab(cuda(b), X, None, tol=1e-10, max_iter=20)
    assert rc == 0 and st[0]["iters"] == 1 and st[0]["mvp"] == 1
    assert st[0]["rel_res"] == 0.0 and st[0]["true_rel_res"] == 0.0
    assert np.array_equal(host(X), b)
    op.close()


@pytest.mark.parametrize("bits", [32, 16])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 16, 16, 10)])
def test_zero_residual_is_zero_in_low_precision(wdl, dims, bits):
    op = wdl.WilsonOperator(dims, cuda(L.gauge_field(dims, 0.5, 32)), 0.0)
    op.set_mixed_storage(bits)
    b = np.zeros((1, op.n), dtype=np.complex128)
    b[0, 5] = 1.0
    X = cuda(np.zeros_like(b))
    rc, st = op.dbicgstab_mixed(cuda(b), X, None, tol=1e-10, max_iter=20)
    assert rc == 0 and st[0]["iters"] == 1 and st[0]["mvp"] == 1
    assert st[0]["true_rel_res"] == 0.0
    assert np.array_equal(host(X), b)
    op.close()
