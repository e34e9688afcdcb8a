"""Labels and fields of the brick-wise phi^4 clusters against the oracle: sides
below, at and just past a brick's in every direction (8 x 4 x 4 x 2 below 2^20
sites, 16 x 8 x 8 x 4 from there), fields from almost no bonds to one
lattice-spanning cluster, and bonds next to the binary32 test's limits."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


def field(L, scale, seed):
    rng = np.random.default_rng(seed)
    return scale * (rng.normal(size=(L, L, L, L, 4)) + rng.normal(size=4))


@pytest.mark.parametrize("L", [2, 4, 7, 8, 9, 16, 17])
@pytest.mark.parametrize("scale", [0.2, 1.0, 5.0])
def test_labels_and_update(sw, L, scale):
    kappa, seed, t = 0.304, 11 + L, 7
    phi = field(L, scale, L)
    with sw.Phi4(L, kappa, seed) as f:
        f.set_field(phi, t)
        lab = f.labels()
        r = oracle.phi4_direction(seed, t)
        want, _ = oracle.phi4_labels(oracle.phi4_bonds(phi, kappa, seed, t, r))
        assert np.array_equal(lab, want)
        f.sweep(2)
        assert np.array_equal(f.field(), oracle.phi4_run(L, kappa, seed, 2, phi=phi, t0=t)[0])


@pytest.mark.parametrize("L", [32, 33])
def test_large_bricks(sw, L):
    kappa, seed, t = 0.304, 3, 1
    phi = field(L, 1.0, L)
    with sw.Phi4(L, kappa, seed) as f:
        f.set_field(phi, t)
        r = oracle.phi4_direction(seed, t)
        want, _ = oracle.phi4_labels(oracle.phi4_bonds(phi, kappa, seed, t, r))
        assert np.array_equal(f.labels(), want)
        f.sweep(1)
        assert np.array_equal(f.field(), oracle.phi4_run(L, kappa, seed, 1, phi=phi, t0=t)[0])


@pytest.mark.parametrize("exponents", [(-70, 70), (-50, 50), (-140, 5), (4, 6)])
def test_mixed_magnitudes(sw, exponents):
    # projections below 2^-60, beyond binary32's range, and z far past 40
    L, kappa, seed = 6, 0.304, 9
    rng = np.random.default_rng(17)
    phi = np.ldexp(rng.normal(size=(L, L, L, L, 4)), rng.integers(*exponents, size=(L, L, L, L, 1)))
    with sw.Phi4(L, kappa, seed) as f:
        f.set_field(phi, 0)
        f.sweep(3)
        assert np.array_equal(f.field(), oracle.phi4_run(L, kappa, seed, 3, phi=phi, t0=0)[0])
