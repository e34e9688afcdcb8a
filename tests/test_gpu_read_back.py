"""Reads of a trace: stretches of every kind of length around the pinned page
they pass through (2 words a sweep, 4095 words to a page) against the oracle."""
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


def test_stretches(sw):
    L, beta, seed, n = 6, 0.4, 3, 4200
    _, want_E, want_M, _ = oracle.run(L, beta, seed, n)
    with sw.Lattice(L, beta, seed) as lat:
        lat.sweep(n)
        b = sw.sw_batch_create([L], [beta], [seed])
        try:
            sw.sw_batch_sweep(b, n)
            for first, count in [(0, n), (0, 0), (n, 0), (n - 1, 1), (1, 64), (7, 2047), (7, 2048), (3, 2049)]:
                for E, M in (lat.observables(first, count), sw.sw_batch_observables(b, 0, first, count)):
                    assert np.array_equal(E, want_E[first:first + count]), (first, count)
                    assert np.array_equal(M, want_M[first:first + count]), (first, count)
        finally:
            sw.sw_batch_destroy(b)
