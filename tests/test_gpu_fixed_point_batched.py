"""The batched fixed-point product (wilson_fx_kernel) on lattices whose site
counts end inside, at and just past a warp's 16 sites, a tile's 32 and a block's
64: as many systems as send them past the few-site form (21504 sites x systems
with an odd extent, 14336 without).  Against the oracle, with the bar of
test_gpu_fixed_point: 64 units of 2^-53 of the largest entry around a site."""
import numpy as np
import pytest

from inputs import lattice as L
from oracle import dirac

from .test_gpu_fixed_point import _apply, _local_max, wdl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs", [((17, 1, 1, 1), 1270), ((31, 1, 1, 1), 700), ((43, 3, 1, 1), 168),
                                       ((8, 4, 4, 1), 170), ((2, 2, 2, 4), 700), ((1, 1, 1, 1), 21600)])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("spread", [0.0, 6.0, 40.0])
def test_batched_edges(wdl, dims, nrhs, dagger, spread):  # noqa: F811
    rng = np.random.Generator(np.random.PCG64(17))
    U = L.gauge_field(dims, 0.9, 41)
    psi = L.gaussian_spinor(dims, 42, nrhs=nrhs)
    psi = psi * 10.0 ** rng.uniform(-spread, spread, size=psi.shape[:2])[:, :, None, None]
    psi[:, 0] = 0.0
    got = _apply(wdl, dims, U, psi, 0.14, 0.07, dagger)
    f = dirac.apply_A_dagger if dagger else dirac.apply_A
    for r in sorted({0, 1, 2, nrhs // 2, nrhs - 1}):
        bound = 64 * 2.0 ** -53 * _local_max(psi[r], dims)
        assert np.all(np.abs(got[r] - f(U, psi[r], dims, 0.14, 0.07)).max(axis=(-1, -2)) <= bound)
