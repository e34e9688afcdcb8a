"""Rows off 16-byte boundaries on the tiled path, bit for bit against the
oracle: every residue of the side mod 16 (row words straddle two or three
16-byte windows, stores start on every byte of a 4-byte word, Philox pairs
straddle rows on odd sides) with a last tile one column to one word wide, the
rows at the two ends of the lattice's memory included."""
import os

import numpy as np
import pytest

import oracle
from workloads import random_spins

pytestmark = pytest.mark.gpu

BETA_C = 0.44068679


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


@pytest.fixture()
def tiled(monkeypatch):
    monkeypatch.setenv("SW_TILE_SHAPE", "6")


@pytest.mark.parametrize("L", [5, 31] + list(range(129, 146)) + [160, 162, 191])
def test_ising_rows(sw, tiled, L):
    seed, n = 40 + L, 4
    s0 = random_spins(L, seed=L)
    with sw.Lattice(L, BETA_C, seed) as lat:
        lat.set_state(s0, 7)
        want_lab, _ = oracle.labels(oracle.bonds(s0, seed, 7, oracle.threshold(BETA_C)))
        assert np.array_equal(lat.labels(), want_lab)
        lat.sweep(n)  # the fused launches
        want_s, want_E, want_M, _ = oracle.run(L, BETA_C, seed, n, spins=s0, t0=7)
        E, M = lat.observables(7, n)
        assert np.array_equal(E, want_E) and np.array_equal(M, want_M)
        assert np.array_equal(lat.spins(), want_s)


@pytest.mark.parametrize("L", [5, 31] + list(range(129, 146)) + [160, 162, 191])
def test_potts_rows(sw, L):
    q, beta, seed, n = 4, 1.1, 50 + L, 4
    with sw.Potts(L, q, beta, seed) as p:
        p.sweep(n)
        want_s, want_E, want_M = oracle.potts_run(L, q, beta, seed, n)
        E, M = p.observables(0, n)
        assert np.array_equal(E, want_E) and np.array_equal(M, want_M)
        assert np.array_equal(p.states(), want_s)
