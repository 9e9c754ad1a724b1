"""Entries far below their neighbours keep FP64's precision: the fixed-point
kernels share exponents over sites, chunks and tiles, and have to fall back to
FP64 where a result rests on entries that the shared exponent does not hold.

Fields: (colours) links that are diagonal in colour and colours of 1, 2^-40 and
2^-80, which the operator never mixes; (point) one site 1e20 above the others
with a single spin, which does not reach every spin of its neighbours.

Bar of an operator product, component by component: FP64 leaves at most 64
units of 2^-53 times the sum of the magnitudes of the terms that reach the
component (48 products, their sums and projections: at most some 60 roundings
of partial sums no larger than it; in practice a few units), per half hop for
the Schur operator, so 128.  Exact zeros stay zero.
"""
import numpy as np
import pytest

from inputs import lattice as L
from oracle import dirac, evenodd

from .gpu_util import cuda, host

pytestmark = pytest.mark.gpu

SCALE = 2.0 ** np.array([0.0, -40.0, -80.0])


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


def _links(dims, kind):
    if kind == "point":
        return L.gauge_field(dims, 0.9, 21)
    rng = np.random.Generator(np.random.PCG64(22))
    ph = np.exp(2j * np.pi * rng.uniform(size=(L.volume(dims), 4, 3)))
    U = np.zeros((L.volume(dims), 4, 3, 3), dtype=np.complex128)
    for c in range(3):
        U[:, :, c, c] = ph[:, :, c]
    return U


def _field(dims, kind, nrhs):
    psi = L.gaussian_spinor(dims, 23, nrhs=nrhs).reshape(nrhs, -1, 4, 3)
    if kind == "colours":
        return psi * SCALE
    p = psi.copy()
    for r in range(nrhs):
        at = (5 * r) % p.shape[1]
        p[r, at] = 0.0
        p[r, at, r % 4] = 1e20
    return p


def _hop_abs(U, a, dims):
    """sum over the hops of |U| (|psi_s| + |psi_partner|): the terms' magnitudes."""
    n = dims[::-1]
    v = L.volume(dims)
    aU = np.abs(U)
    out = np.zeros((v, 4, 3))
    site = np.arange(v).reshape(n)
    for mu in range(4):
        part = [3, 2, 1, 0] if mu < 2 else [2, 3, 0, 1]
        h = a + a[:, part]
        up = np.roll(site, -1, 3 - mu).reshape(-1)
        dn = np.roll(site, 1, 3 - mu).reshape(-1)
        out += np.einsum("sab,sib->sia", aU[:, mu], h[up])
        out += np.einsum("sba,sib->sia", aU[dn, mu], h[dn])
    return out


@pytest.mark.parametrize("dims,nrhs", [((4, 4, 4, 4), 1), ((3, 5, 7, 2), 3), ((8, 4, 4, 8), 12), ((9, 7, 5, 11), 4),
                                       ((8, 4, 4, 8), 16), ((9, 7, 5, 11), 7)])   # the batched form
@pytest.mark.parametrize("kind", ["colours", "point"])
@pytest.mark.parametrize("dagger,mu", [(False, 0.0), (True, 0.07)])
def test_product(wdl, dims, nrhs, kind, dagger, mu):
    import torch
    U, psi = _links(dims, kind), _field(dims, kind, nrhs)
    op = wdl.WilsonOperator(dims, cuda(U), 0.14, mu)
    out = torch.empty(psi.size, dtype=torch.complex128, device="cuda:0")
    op.apply(cuda(psi), out, dagger=dagger)
    got = host(out).reshape(psi.shape)
    op.close()
    f = dirac.apply_A_dagger if dagger else dirac.apply_A
    for r in range(nrhs):
        ref = f(U, psi[r], dims, 0.14, mu)
        a = np.abs(psi[r])
        bound = 64 * 2.0 ** -53 * ((1 + mu) * a + 0.14 * _hop_abs(U, a, dims))
        assert np.all(np.abs(got[r] - ref) <= bound)


@pytest.mark.parametrize("dims,nrhs", [((4, 4, 4, 4), 1), ((2, 6, 4, 8), 5), ((8, 8, 4, 6), 3)])
@pytest.mark.parametrize("kind", ["colours", "point"])
@pytest.mark.parametrize("dagger,mu", [(False, 0.0), (True, 0.07), (False, 0.07)])
def test_schur_product(wdl, dims, nrhs, kind, dagger, mu):
    import torch
    U = _links(dims, kind)
    v = L.volume(dims)
    half = np.ascontiguousarray(_field(dims, kind, nrhs)[:, : v // 2])
    op = wdl.WilsonOperator(dims, cuda(U), 0.14, mu)
    op.set_operator(True)
    out = torch.empty(half.size, dtype=torch.complex128, device="cuda:0")
    op.apply(cuda(half), out, dagger=dagger)
    got = host(out).reshape(half.shape)
    op.close()
    s = np.indices(dims[::-1]).sum(0).reshape(-1) % 2 == 0
    g5 = lambda z: dirac.gamma5(z.reshape(-1, 4, 3))
    for r in range(nrhs):
        if dagger:
            ref = g5(evenodd.schur_apply(U, dims, 0.14, -mu, g5(half[r]).ravel()))
        else:
            ref = evenodd.schur_apply(U, dims, 0.14, mu, half[r].ravel())
        full = np.zeros((v, 4, 3))
        full[s] = np.abs(half[r])
        two = _hop_abs(U, _hop_abs(U, full, dims), dims)[s] * (1 + mu)
        bound = 128 * 2.0 ** -53 * ((1 + mu) * np.abs(half[r]) + 0.14 ** 2 * two)
        assert np.all(np.abs(got[r] - ref.reshape(-1, 4, 3)) <= bound)


@pytest.mark.parametrize("dims,nrhs", [((4, 4, 4, 4), 1), ((8, 8, 8, 16), 2), ((16, 16, 16, 10), 1)])
@pytest.mark.parametrize("even_odd", [False, True])
def test_bicgstab_carries_every_colour(wdl, dims, nrhs, even_odd):
    """Colours with the same links and source up to a power of two have the same
    solution up to it, also step by step: FP64 arithmetic scales exactly.  Three
    steps at kappa = 0.1 of some six vector operations, each within 64 units of
    2^-53 in the norm: 1.3e-13, and a factor of 8 for what the steps amplify."""
    ph = _links(dims, "colours")
    for c in (1, 2):
        ph[:, :, c, c] = ph[:, :, 0, 0]
    op = wdl.WilsonOperator(dims, cuda(ph), 0.1)
    op.set_operator(even_odd)
    b = L.gaussian_spinor(dims, 24, nrhs=nrhs).reshape(nrhs, -1, 4, 3)[:, : op.op_n // 12]
    b = b[..., :1] * SCALE
    X = cuda(np.zeros_like(b))
    op.dbicgstab(cuda(b).reshape(-1), X.reshape(-1), None, tol=1e-15, max_iter=3)
    x = host(X) / SCALE
    op.close()
    for c in (1, 2):
        assert np.linalg.norm(x[..., c] - x[..., 0]) <= 1e-12 * np.linalg.norm(x[..., 0])


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (5, 13, 3, 2), (8, 8, 8, 4)])
@pytest.mark.parametrize("m,k", [(12, 0), (40, 12)])
def test_gmresdr_carries_every_colour(wdl, dims, m, k):
    """The same through the Gram-Schmidt products: a basis vector's colours stay
    equal up to the power of two, and so does the solution; 1e-11 as for two
    runs that differ by rounding (condition of the least squares below 1e3)."""
    import torch
    ph = _links(dims, "colours")
    for c in (1, 2):
        ph[:, :, c, c] = ph[:, :, 0, 0]
    op = wdl.WilsonOperator(dims, cuda(ph), 0.12)
    b = (L.gaussian_spinor(dims, 25)[..., :1] * SCALE).reshape(-1)
    X = cuda(np.zeros_like(b))
    V = torch.zeros(max(k, 1) * b.size, dtype=torch.complex128, device="cuda:0")
    op.gmresdr(cuda(b), X, m, k, 1e-14, m + (m - k if k else 0), V_out=V if k else None)
    x = host(X).reshape(-1, 3) / SCALE
    op.close()
    for c in (1, 2):
        assert np.linalg.norm(x[:, c] - x[:, 0]) <= 1e-11 * np.linalg.norm(x[:, 0])
    if k:
        w = host(V).reshape(-1, 3) / SCALE
        for c in (1, 2):
            assert np.linalg.norm(w[:, c] - w[:, 0]) <= 1e-11 * np.linalg.norm(w[:, 0])
