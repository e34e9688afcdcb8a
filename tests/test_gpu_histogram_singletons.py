"""Cluster statistics where one bin takes every site: at beta = 0 each site is
its own cluster, so a thread of phase 3 meets as many roots as its strip has
sites (up to 8 rows of 32), all of size 1; and next to it, with few bonds."""
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


@pytest.mark.parametrize("shape", range(10))
@pytest.mark.parametrize("beta", [0.0, 0.02, 0.2])
def test_every_shape(sw, shape, beta, monkeypatch):
    monkeypatch.setenv("SW_TILE_SHAPE", str(shape))
    L, seed, n = 389, 4, 2  # tiles with whole strips inside, and ragged ones
    _, want_E, _, want = oracle.run(L, beta, seed, n, hist=True)
    with sw.Lattice(L, beta, seed) as lat:
        lat.histogram(True)
        lat.sweep(n)
        assert np.array_equal(lat.histograms(0, n), want)
        assert np.array_equal(lat.observables(0, n)[0], want_E)
    if beta == 0.0:
        assert (want[:, 0] == L * L).all() and (want[:, 2] == L * L).all()
