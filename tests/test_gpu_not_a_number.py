"""NaN and infinities that reach the small dense problems: an error or a result,
never an index out of range.  The LU of the projected matrix (a column of NaN has
no pivot), the order of harmonic Ritz values that are NaN, and the basis of a
GMRES-DR solve that ended before it had k vectors."""
import numpy as np
import pytest

from inputs import lattice as L

from .gpu_util import cuda, host, oracle_ops

pytestmark = pytest.mark.gpu

SINGULAR = 4   # WD_SINGULAR_PROJECTION


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


def _operator(wdl, dims):
    return wdl.WilsonOperator(dims, cuda(L.gauge_field(dims, 0.5, 71)), 0.12)


@pytest.mark.parametrize("k", [1, 2, 33])
def test_deflation_space_with_nan_is_singular(wdl, k):
    op = _operator(wdl, (4, 4, 2, 2))
    rng = np.random.Generator(np.random.PCG64(72))
    V = rng.normal(size=(k, op.n)) + 1j * rng.normal(size=(k, op.n))
    V[k // 2, 5] = np.nan
    with pytest.raises(wdl.WdError) as e:
        op.deflation(cuda(V), k)
    assert e.value.status == SINGULAR
    V[k // 2, 5] = 1.0
    d = op.deflation(cuda(V), k)          # the handle is as good as before
    d.close()
    op.close()


def test_vectors_after_a_lucky_breakdown_are_zero(wdl):
    """A source in an invariant subspace of two vectors (unit links, momenta 0
    and (pi, 0, 0, 0)): the basis ends there, the other vectors are zero."""
    import torch
    dims = (4, 2, 2, 2)
    v = L.volume(dims)
    op = wdl.WilsonOperator(dims, cuda(L.unit_gauge_field(dims)), 0.1)
    b = np.zeros((v, 4, 3), dtype=np.complex128)
    b[:, 0, 0] = 1.0
    b[:, 0, 1] = (-1.0) ** (np.arange(v) % 4)
    x = cuda(np.zeros(op.n, dtype=np.complex128))
    V = torch.full((6 * op.n,), float("nan"), dtype=torch.complex128, device="cuda:0")
    rc, st, hbar, theta = op.gmresdr(cuda(b.ravel()), x, 12, 6, 1e-12, 100, V_out=V)
    assert rc == 0 and st["mvp"] == 2
    w = host(V).reshape(6, -1)
    assert np.all(np.isfinite(w)) and not w[2:].any() and w[:2].any()
    assert np.all(np.isfinite(hbar)) and np.all(np.isfinite(theta))
    op.close()


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_sources_that_are_not_finite(wdl, value):
    import torch
    dims = (4, 4, 2, 2)
    op = _operator(wdl, dims)
    b = L.gaussian_spinor(dims, 73).ravel()
    bad = b.copy()
    bad[7] = value
    for m, k in ((8, 0), (12, 5)):
        x = cuda(np.zeros_like(b))
        try:
            rc, st, _, _ = op.gmresdr(cuda(bad), x, m, k, 1e-10, 40)
            assert not st["converged"]
        except wdl.WdError:
            pass                          # the restart's eigenproblem failed
    X = torch.zeros(2, 2, b.size, dtype=torch.complex128, device="cuda:0")
    rc, st = op.multishift(cuda(np.stack([bad, b])), X, [0.1, 0.05], tol=1e-10, max_iter=200)
    assert rc != 0 and not st[0][0]["converged"] and st[0][1]["converged"] and st[1][1]["converged"]
    A, g5 = oracle_ops(L.gauge_field(dims, 0.5, 71), dims, 0.12)
    x = cuda(np.zeros_like(b))
    rc, st, _, _ = op.gmresdr(cuda(b), x, 12, 5, 1e-10, 400)    # the handle is as good as before
    assert rc == 0 and np.linalg.norm(b - A(host(x))) <= 2e-10 * np.linalg.norm(b)
    op.close()
