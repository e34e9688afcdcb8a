"""Bonds of the phi^4 update at couplings and fields near the ends of the
number range (products of order one from a tiny coupling and a large field),
against the oracle."""
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


@pytest.mark.parametrize("log2_kappa", [-147, -140, -127, -100, -68, -67, 0])
@pytest.mark.parametrize("uneven", [False, True])
def test_labels(sw, log2_kappa, uneven):
    L, seed, t = 6, 13, 2
    kappa = 1.37 * 2.0 ** log2_kappa
    rng = np.random.default_rng(-log2_kappa + uneven)
    phi = 2.0 ** (-log2_kappa / 2 - 1) * rng.normal(size=(L, L, L, L, 4))
    if uneven:  # every other site small, its neighbours large: the products stay
        step = 2.0 ** min(50.0, 60.0 + log2_kappa / 2) if log2_kappa > -120 else 2.0 ** 30
        odd = np.indices((L,) * 4).sum(axis=0)[..., None] % 2 == 1
        phi = np.where(odd, phi * step, phi / step)
    r = oracle.phi4_direction(seed, t)
    want, _ = oracle.phi4_labels(oracle.phi4_bonds(phi, kappa, seed, t, r))
    with sw.Phi4(L, kappa, seed) as f:
        f.set_field(phi, t)
        assert np.array_equal(f.labels(), want)
        f.sweep(2)
        assert np.array_equal(f.field(), oracle.phi4_run(L, kappa, seed, 2, phi=phi, t0=t)[0])
