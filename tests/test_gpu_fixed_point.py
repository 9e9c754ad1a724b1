"""The fixed-point hops of the FP64 Wilson operator (wd_apply on SU(3) links)
against the oracle, and against the FP64 kernel that serves every other link
field, where the two could part: tile and block edges, magnitudes that vary
from site to site, zeros, and values that fixed point does not hold.

Bar: each output component is a sum of 48 products per hop direction pair; a
site's slices hold its entries to 2^-57 of its largest, a product leaves out
less than 2^-57 of it, and the sum is rounded once, so the error of a
component is below 16 units of 2^-53 times M, the largest entry among the
site and its neighbours (8 hops x 2 spins x sqrt(3) colours of unit-norm links
bound the sum by 2^5 M; FP64 roundings of sums of that size, at most 2^-53 of
it each, are what the oracle itself leaves: another 2^5 x 48 x 2^-53 M at the
very most, in practice a few units).  The test allows 64 units.
"""
import numpy as np
import pytest

from inputs import lattice as L
from oracle import dirac

from .gpu_util import cuda, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wdl():
    import paper_0710_1988_gb300 as wdl
    wdl.lib()
    return wdl


def _local_max(psi, dims):
    """Largest |re| or |im| among every site and its eight neighbours, (V,)."""
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-1, -2)).reshape(dims[::-1])
    out = m.copy()
    for ax in range(4):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out.reshape(-1)


def _apply(wdl, dims, U, psi, kappa, mu=0.0, dagger=False):
    import torch
    op = wdl.WilsonOperator(dims, cuda(U), kappa, mu)
    out = torch.empty(psi.size, dtype=torch.complex128, device="cuda:0")
    op.apply(cuda(psi), out, dagger=dagger)
    got = host(out).reshape(psi.shape)
    op.close()
    return got


@pytest.mark.parametrize("dims,nrhs", [((13, 9, 7, 15), 1), ((16, 16, 6, 8), 1), ((11, 9, 7, 2), 9),
                                       # the same edges in the form for more than 12288 sites x systems
                                       ((17, 1, 1, 1), 742), ((31, 1, 1, 1), 400), ((43, 3, 1, 1), 98),
                                       ((8, 4, 4, 1), 97), ((2, 2, 2, 4), 400), ((1, 1, 1, 1), 12300),
                                       ((1, 1, 1, 1), 1), ((3, 5, 1, 1), 2), ((4, 4, 1, 1), 1),
                                       ((17, 1, 1, 1), 1), ((31, 1, 1, 1), 1), ((2, 2, 2, 4), 3),
                                       ((11, 3, 1, 1), 1), ((127, 1, 1, 1), 2), ((8, 4, 4, 1), 1),
                                       ((43, 3, 1, 1), 3), ((6, 2, 4, 8), 2), ((9, 7, 5, 3), 4)])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("spread", [0.0, 6.0, 40.0])
def test_edges_and_magnitudes(wdl, dims, nrhs, dagger, spread):
    rng = np.random.Generator(np.random.PCG64(17))
    U = L.gauge_field(dims, 0.9, 41)
    psi = L.gaussian_spinor(dims, 42, nrhs=nrhs)
    psi = psi * 10.0 ** rng.uniform(-spread, spread, size=psi.shape[:2])[:, :, None, None]
    psi[:, 0] = 0.0
    got = _apply(wdl, dims, U, psi, 0.14, 0.07, dagger)
    f = dirac.apply_A_dagger if dagger else dirac.apply_A
    for r in sorted({0, 1 % nrhs, 2 % nrhs, nrhs // 2, nrhs - 1}):
        ref = f(U, psi[r], dims, 0.14, 0.07)
        bound = 64 * 2.0 ** -53 * _local_max(psi[r], dims)
        assert np.all(np.abs(got[r] - ref).max(axis=(-1, -2)) <= bound)


@pytest.mark.parametrize("nrhs", [1, 40])     # few sites in all, and many
def test_values_outside_fixed_point_match_the_fp64_kernel(wdl, nrhs):
    """Infinities, NaN, subnormal and very large entries beside ordinary ones:
    the same finite values, and the same infinities and NaN, as the FP64
    kernel gives (an operator whose only difference is one scaled link, which
    sends it to that kernel, read away from that link)."""
    dims = (6, 4, 4, 4)
    U = L.gauge_field(dims, 0.5, 51)
    U2 = U.copy()
    far = L.volume(dims) - 1
    U2[far, 0] *= 4.0
    psi = L.gaussian_spinor(dims, 52)
    psi[7, 0, 1] = np.inf
    psi[100, 2, 0] = complex(0.0, np.nan)
    psi[150] *= 1e-310
    psi[160] *= 1e300
    psi[170] = 0.0
    psi[171] = 5e-324
    a = _apply(wdl, dims, U, np.stack([psi] * nrhs), 0.14)[-1]
    b = _apply(wdl, dims, U2, np.stack([psi] * nrhs), 0.14)[-1]
    keep = np.ones(L.volume(dims), dtype=bool)
    keep[[far, far - 5]] = False          # the two ends of the scaled x link
    a, b = a[keep], b[keep]
    for x, y in ((a.real, b.real), (a.imag, b.imag)):
        assert np.array_equal(np.isnan(x), np.isnan(y))
        inf = np.isinf(y)
        assert np.array_equal(inf, np.isinf(x)) and np.array_equal(x[inf], y[inf])
    fin = np.isfinite(b)
    clean = psi.copy()
    clean[~np.isfinite(clean)] = 0.0
    bound = np.broadcast_to((64 * 2.0 ** -53 * _local_max(clean, dims))[keep][:, None, None], a.shape)
    assert np.all(np.abs(a[fin] - b[fin]) <= bound[fin])


@pytest.mark.parametrize("scale", [3.0, 1e-3])
def test_links_that_are_not_unitary(wdl, scale):
    dims = (4, 3, 2, 5)
    U = L.gauge_field(dims, 0.5, 61) * scale
    psi = L.gaussian_spinor(dims, 62, nrhs=2)
    got = _apply(wdl, dims, U, psi, 0.13)
    for r in range(2):
        ref = dirac.apply_A(U, psi[r], dims, 0.13)
        assert np.abs(got[r] - ref).max() <= 1e-12 * np.abs(ref).max()


def test_unit_links_are_exact(wdl):
    """Dyadic values on unit links: every product and sum is exact."""
    dims = (4, 2, 2, 3)
    U = L.unit_gauge_field(dims)
    rng = np.random.Generator(np.random.PCG64(71))
    psi = (rng.integers(-64, 65, size=(L.volume(dims), 4, 3))
           + 1j * rng.integers(-64, 65, size=(L.volume(dims), 4, 3))) / 8.0
    assert np.array_equal(_apply(wdl, dims, U, psi, 0.125), dirac.apply_A(U, psi, dims, 0.125))


def _schur(wdl, dims, U, half, kappa, mu=0.0, dagger=False):
    import torch
    op = wdl.WilsonOperator(dims, cuda(U), kappa, mu)
    op.set_operator(True)
    out = torch.empty(half.size, dtype=torch.complex128, device="cuda:0")
    op.apply(cuda(half), out, dagger=dagger)
    got = host(out).reshape(half.shape)
    op.close()
    return got


def _two_hop_max(half, dims):
    """Largest |re| or |im| of the even sites within two hops, at the even sites."""
    v = L.volume(dims)
    full = np.zeros((v, 4, 3), dtype=np.complex128)
    even = _even_sites(dims)
    full[even] = half
    m = _local_max(full, dims)
    return _local_max(np.broadcast_to(m[:, None, None] + 0j, (v, 1, 1)), dims)[even]


def _even_sites(dims):
    s = np.arange(L.volume(dims))
    x, s = s % dims[0], s // dims[0]
    y, s = s % dims[1], s // dims[1]
    z, t = s % dims[2], s // dims[2]
    return (x + y + z + t) % 2 == 0


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((4, 2, 2, 2), 3), ((2, 2, 2, 10), 2),
                                       ((6, 4, 2, 6), 2), ((34, 2, 4, 2), 1), ((8, 8, 2, 4), 3)])
@pytest.mark.parametrize("mu", [0.0, 0.07])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("spread", [0.0, 20.0])
def test_schur_edges_and_magnitudes(wdl, dims, nrhs, mu, dagger, spread):
    """Each half hop leaves 64 units of 2^-53 of its largest entry and grows
    entries by at most 2^5: 2^12 units of kappa^2 M over two hops, 64 of M."""
    from oracle import evenodd
    rng = np.random.Generator(np.random.PCG64(18))
    U = L.gauge_field(dims, 0.9, 43)
    half = L.gaussian_spinor(dims, 44, nrhs=nrhs)[:, : L.volume(dims) // 2]
    half = half * 10.0 ** rng.uniform(-spread, spread, size=half.shape[:2])[:, :, None, None]
    half[:, 0] = 0.0
    got = _schur(wdl, dims, U, half, 0.14, mu, dagger)
    g5 = lambda z: dirac.gamma5(z.reshape(-1, 4, 3))
    for r in range(nrhs):
        if dagger:
            ref = g5(evenodd.schur_apply(U, dims, 0.14, -mu, g5(half[r]).ravel()))
        else:
            ref = evenodd.schur_apply(U, dims, 0.14, mu, half[r].ravel())
        ref = ref.reshape(half[r].shape)
        bound = (4096 * 0.14 ** 2 + 64) * 2.0 ** -53 * _two_hop_max(half[r], dims)
        assert np.all(np.abs(got[r] - ref).max(axis=(-1, -2)) <= bound)


@pytest.mark.parametrize("mu", [0.0, 0.07])
def test_schur_values_outside_fixed_point_match_the_fp64_kernel(wdl, mu):
    """As for the full operator; the scaled link reaches two hops."""
    dims = (8, 4, 4, 8)
    v = L.volume(dims)
    U = L.gauge_field(dims, 0.5, 53)
    U2 = U.copy()
    far = v - 1
    U2[far, 0] *= 4.0
    half = L.gaussian_spinor(dims, 54)[: v // 2]
    half[7, 0, 1] = np.inf
    half[100, 2, 0] = complex(0.0, np.nan)
    half[150] *= 1e-310
    half[160] *= 1e300
    half[170] = 0.0
    half[171] = 5e-324
    a, b = _schur(wdl, dims, U, half, 0.14, mu), _schur(wdl, dims, U2, half, 0.14, mu)
    hit = np.zeros((v, 1, 1), dtype=np.complex128)
    hit[[far, far - 7]] = 1.0             # the ends of the scaled x link
    even = _even_sites(dims)
    keep = _local_max(hit, dims)[even] == 0.0
    for x, y in ((a.real[keep], b.real[keep]), (a.imag[keep], b.imag[keep])):
        assert np.array_equal(np.isnan(x), np.isnan(y))
        inf = np.isinf(y)
        assert np.array_equal(inf, np.isinf(x)) and np.array_equal(x[inf], y[inf])
    clean = half.copy()
    clean[~np.isfinite(clean)] = 0.0
    bound = ((4096 * 0.14 ** 2 + 64) * 2.0 ** -53 * _two_hop_max(clean, dims))[keep][:, None, None]
    fin = np.isfinite(b[keep])
    assert np.all(np.abs(a[keep] - b[keep])[fin] <= np.broadcast_to(bound, a[keep].shape)[fin])
