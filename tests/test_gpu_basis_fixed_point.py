"""The fixed-point Gram-Schmidt products of GMRES-DR (fx_basis.cu) where they
can go wrong: vectors that end inside, at and just past a chunk of 64 sites,
basis sizes around a dot block's 16 vectors and an update's 32-vector fold,
sources whose magnitudes vary from site to site, and a chunk whose entries
fixed point does not hold (it takes FP64).

Against the oracle's GMRES-DR (FP64, classical Gram-Schmidt twice as well).
Bars: two backward stable runs differ by rounding times the condition of the
m-step least squares problem, below 1e3 for these operators (sigma_max /
sigma_min of A below 1e2): 1e3 * m * 2^-53 < 1e-11 in x, and in theta as long as
the cycles have not reached rounding level (the harmonic Ritz values of a
residual of 1e-10 are determined to 1e-6 only: compared when the residual is
above 1e-7); the least-squares residual is the true one to 1e-12 because
A V_m = V_{m+1} Hbar_m holds to rounding; the basis is orthonormal to
m * 2^-53 * 8 < 1e-13; the deflated start of a next source is compared with the
same projection formed here from the basis returned: 1e-9 allows for a
condition of G up to 1e6.
"""
import numpy as np
import pytest

from inputs import lattice as L
from oracle import krylov

from .gpu_util import cuda, host, oracle_ops

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


def _source(dims, kind):
    b = L.gaussian_spinor(dims, 92)
    if kind == "spread":
        rng = np.random.Generator(np.random.PCG64(93))
        b *= 10.0 ** rng.uniform(-6.0, 0.0, size=b.shape[0])[:, None, None]
    elif kind == "point":
        b[1:] = 0.0
    elif kind == "tiny_chunk":
        b[:64] *= 1e-260
    return b.ravel()


@pytest.mark.parametrize("dims", [(3, 3, 7, 1), (4, 4, 4, 1), (5, 13, 1, 1), (11, 7, 5, 3)])
@pytest.mark.parametrize("m,k", [(15, 0), (16, 5), (17, 4), (33, 16), (70, 20)])
@pytest.mark.parametrize("kind", ["plain", "spread", "point", "tiny_chunk"])
def test_cycles_match_oracle(wdl, dims, m, k, kind):
    import torch
    if kind == "tiny_chunk" and L.volume(dims) <= 64:
        pytest.skip("one chunk")
    U = L.gauge_field(dims, 0.5, 91)
    kappa = 0.12
    A, g5 = oracle_ops(U, dims, kappa)
    b = _source(dims, kind)
    budget = m + (m - k)
    gd = krylov.gmresdr(A, b, m, k, tol=1e-14, max_mv=budget)
    op = wdl.WilsonOperator(dims, cuda(U), kappa)
    x = cuda(np.zeros_like(b))
    V = torch.zeros(max(k, 1) * b.size, dtype=torch.complex128, device="cuda:0")
    rc, st, hbar, theta = op.gmresdr(cuda(b), x, m, k, 1e-14, budget, V_out=V if k else None)
    assert st["mvp"] == gd.stats.mvp
    assert np.linalg.norm(host(x) - gd.x) <= 1e-11 * np.linalg.norm(gd.x)
    assert abs(st["rel_res"] - st["true_rel_res"]) <= 1e-12
    if k and gd.stats.rel_res > 1e-7:
        assert np.abs(np.sort(np.abs(theta)) - np.sort(np.abs(gd.theta))).max() <= 1e-11 * np.abs(gd.theta).max()
    if k:
        Vh = host(V).reshape(k, -1)
        assert np.abs(Vh.conj() @ Vh.T - np.eye(k)).max() <= 1e-13
        # the projection of a next source (G = V^dagger gamma5 A V in fixed point)
        b2 = L.gaussian_spinor(dims, 94).ravel()
        defl = op.deflation(V, k)
        X = cuda(np.zeros_like(b2))
        op.dbicgstab(cuda(b2), X, defl, tol=1e-14, max_iter=1)
        Ug = np.stack([g5(v) for v in Vh])
        y, _, AV = krylov.lr_projection(A, Vh, Ug, b2)
        x1, r = Vh.T @ y, b2 - AV.T @ y
        ar = A(r)
        alpha = np.vdot(r, r) / np.vdot(r, ar)
        s = r - alpha * ar
        t = A(s)
        ref = x1 + alpha * r + np.vdot(t, s) / np.vdot(t, t) * s
        assert np.linalg.norm(host(X) - ref) <= 1e-9 * np.linalg.norm(ref)
        defl.close()
    op.close()


@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (17, 1, 1, 1), (3, 3, 7, 1), (4, 4, 4, 1), (5, 13, 1, 1),
                                  (11, 7, 5, 3)])
@pytest.mark.parametrize("kind", ["plain", "spread", "point", "tiny_chunk"])
@pytest.mark.parametrize("iters", [1, 3])
def test_bicgstab_steps_match_oracle(wdl, dims, kind, iters):
    """Whole BiCGStab iterations (fx_stream.cu: updates and dots on tiles of 16
    sites) from the same start.  Three steps at kappa = 0.1, where A is within
    0.8 of the unit matrix, amplify rounding by less than 1e3: 1e-12.  A system
    whose rho vanishes to rounding (a point source far from its own images:
    the oracle breaks down at its second step) has no such bar and is left out."""
    U = L.gauge_field(dims, 0.5, 95)
    A, _ = oracle_ops(U, dims, 0.1)
    b = _source(dims, kind)
    if kind == "tiny_chunk":
        b = L.gaussian_spinor(dims, 92).reshape(-1, 12)
        b[16:48] *= 1e-260               # two tiles that fixed point does not hold
        b = b.ravel()
    batch = np.stack([b, L.gaussian_spinor(dims, 96).ravel()])
    op = wdl.WilsonOperator(dims, cuda(U), 0.1)
    X = cuda(np.zeros_like(batch))
    op.dbicgstab(cuda(batch), X, None, tol=1e-15, max_iter=iters)
    for got, rhs in zip(host(X), batch):
        ref, so = krylov.bicgstab(A, rhs, tol=1e-15, max_iter=iters)
        if so.breakdown:
            continue
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    op.close()


@pytest.mark.parametrize("dims", [(8, 8, 16, 1), (43, 8, 3, 1), (10, 10, 10, 6), (26, 16, 16, 10)])
@pytest.mark.parametrize("scale", [1.0, 1e-130])
def test_scalar_steps_over_partials(wdl, dims, scale):
    """The dots' block partials (bicg_fin.cuh): 128, 129, 750 and 1040 of them,
    in fixed point and, for squares below its range, in FP64.  Two steps at
    kappa = 0.1: 1e-12, as above."""
    U = L.gauge_field(dims, 0.5, 97)
    A, _ = oracle_ops(U, dims, 0.1)
    b = L.gaussian_spinor(dims, 98).ravel()
    ref, _ = krylov.bicgstab(A, b, tol=1e-15, max_iter=2)
    op = wdl.WilsonOperator(dims, cuda(U), 0.1)
    X = cuda(np.zeros_like(b)[None])
    op.dbicgstab(cuda(scale * b[None]), X, None, tol=1e-15, max_iter=2)
    assert np.linalg.norm(host(X)[0] / scale - ref) <= 1e-12 * np.linalg.norm(ref)
    op.close()
